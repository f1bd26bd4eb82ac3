"""Shapes the library picks by batch size: transforms (forward and inverse) and
products on both sides of every limit give the oracle's words, on batches whose
limbs all differ, with one prime and with three."""
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
    edges = [1, 8, sms // 8, (sms - 8) // 4, limit * 3 // 4, limit]
    edges = sorted({c + d for c in edges for d in (0, 1)} - {0})
    r = Rng(log_n)
    for limbs in (1, 3):              # limb i of the batch uses prime i mod limbs
        qs = he.primes_generate(60, 2 * N, limbs)
        t = he.NttTables(N, qs)
        counts = [c // limbs for c in edges if c % limbs == 0]
        if not counts:
            continue
        x, y = (np.stack([r.uniform_limbs(qs, N) for _ in range(counts[-1])]) for _ in range(2))
        fwd = np.stack([oracle.ntt_fwd(p, qs) for p in x])
        inv = np.stack([oracle.ntt_inv(p, qs) for p in x])
        product = np.stack([oracle.negacyclic_mul(p, q, qs) for p, q in zip(x, y)])
        for count in counts:
            for f, want in ((he.ntt_fwd, fwd), (he.ntt_inv, inv)):
                d = dev(x[:count])
                f(d, N, limbs, count, t)
                assert np.array_equal(host(d), want[:count]), (limbs, count)
            c = empty(count, limbs, N)
            he.negacyclic_mul(c, dev(x[:count]), dev(y[:count]), N, limbs, count, t)
            assert np.array_equal(host(c), product[:count]), (limbs, count)


@pytest.mark.parametrize("log_n", [12, 15, 16])
def test_auto_shape_fused_modup(log_n):
    """The product at minimum scratch, on both sides of the fused mod-up's limit."""
    N, n = 1 << log_n, 2
    data, P = he.chain_primes(N, [50] * n, 60)
    r = Rng(log_n)
    evk = np.stack([np.stack([r.uniform_limbs(data + [P], N) for _ in range(2)]) for _ in range(n)])
    limit = torch.cuda.get_device_properties(0).multi_processor_count * 4096 // N // (n + 1)
    ca, cb = (np.stack([np.stack([r.uniform_limbs(data, N) for _ in range(2)]) for _ in range(limit + 1)])
              for _ in range(2))
    want = np.stack([oracle.mul_relin_rescale(a, b, evk, data, P, n - 1) for a, b in zip(ca, cb)])
    ctx = he.Context(N, data, P)
    key = he.RelinKey(ctx, evk)
    for count in (limit, limit + 1):
        out = empty(count, 2, n - 1, N)
        he.mul_relin_rescale(out, dev(ca[:count]), dev(cb[:count]), count, key, ctx, n - 1,
                             empty(ctx.mrr_scratch_bytes(n - 1, count, 0) // 8))
        assert np.array_equal(host(out), want[:count]), count
