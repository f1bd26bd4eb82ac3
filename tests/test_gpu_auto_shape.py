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

from tests.gpu_util import dev, host  # noqa: E402


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
