"""Shapes the library picks by batch size: transforms and products on both sides
of the small-batch limit give the same words as the oracle and as a fixed
shape, forward, inverse and back."""
import numpy as np
import pytest

import oracle
from paper_2109_14704_gb300 import he
from paper_2109_14704_gb300.synth import Rng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.gpu_util import dev, empty, host  # noqa: E402


@pytest.mark.parametrize("log_n", range(10, 17))
def test_auto_shape_sides(log_n):
    N = 1 << log_n
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    limit = sms * 4096 // N
    qs = he.primes_generate(60, 2 * N, 1)
    t = he.NttTables(N, qs)
    r = Rng(log_n)
    row = r.uniform_limbs(qs, N)
    want_f, want_i = oracle.ntt_fwd(row, qs)[0], oracle.ntt_inv(row, qs)[0]
    edges = [1, 8, sms // 8, limit * 3 // 4, limit]
    for count in sorted({c + d for c in edges for d in (0, 1)} - {0}):
        for f, want in ((he.ntt_fwd, want_f), (he.ntt_inv, want_i)):
            d = dev(row).repeat(count, 1).contiguous()
            f(d, N, 1, count, t)
            got = host(d)
            assert np.array_equal(got[0], want) and (got == want).all(), count
        a = dev(row).repeat(count, 1).contiguous()
        c = torch.empty_like(a)
        he.negacyclic_mul(c, a, a, N, 1, count, t)
        if count == 1:
            want_c = oracle.negacyclic_mul(row, row, qs)[0]
        assert (host(c) == want_c).all(), count


@pytest.mark.parametrize("log_n", [12, 15, 16])
def test_auto_shape_fused_modup(log_n):
    """The product at minimum scratch, on both sides of the fused mod-up's limit."""
    N, n = 1 << log_n, 2
    data, P = he.chain_primes(N, [50] * n, 60)
    r = Rng(log_n)
    evk = np.stack([np.stack([r.uniform_limbs(data + [P], N) for _ in range(2)]) for _ in range(n)])
    ct = np.stack([r.uniform_limbs(data, N) for _ in range(2)])
    want = oracle.mul_relin_rescale(ct, ct, evk, data, P, n - 1)
    ctx = he.Context(N, data, P)
    key = he.RelinKey(ctx, evk)
    limit = torch.cuda.get_device_properties(0).multi_processor_count * 4096 // N // (n + 1)
    for count in (limit, limit + 1):
        a = dev(ct[None]).repeat(count, 1, 1, 1).contiguous()
        out = empty(count, 2, n - 1, N)
        he.mul_relin_rescale(out, a, a, count, key, ctx, n - 1, empty(ctx.mrr_scratch_bytes(n - 1, count, 0) // 8))
        assert (host(out) == want).all(), count
