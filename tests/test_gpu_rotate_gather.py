"""Rotation gathered on the loads of the key switch (no permuted copy): every
kind of Galois element, the per-tile, tiled and fused multiply-accumulates, 8
and 16 words a thread, in place, bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2109_14704_gb300 import he
from paper_2109_14704_gb300.synth import Rng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.gpu_util import dev, empty, host  # noqa: E402


@pytest.mark.parametrize("N,n,count,log_e,minimum", [(1024, 4, 1, 4, True), (1024, 4, 1, 4, False),
                                                     (2048, 3, 9, 4, False), (8192, 2, 2, 3, False)])
@pytest.mark.parametrize("elt", ["1", "3", "5^k", "2N-1"])
def test_rotate_gather(N, n, count, log_e, minimum, elt):
    data, P = he.chain_primes(N, [60] + [50] * (n - 1), 60)
    r = Rng(N + n + count)
    evk = np.stack([np.stack([r.uniform_limbs(data + [P], N) for _ in range(2)]) for _ in range(n)])
    ct = np.stack([np.stack([r.uniform_limbs(data, N) for _ in range(2)]) for _ in range(count)])
    g = {"1": 1, "3": 3, "5^k": pow(5, N // 3, 2 * N), "2N-1": 2 * N - 1}[elt]
    ctx = he.Context(N, data, P)
    ctx.set_eval_shape(log_e)
    key = he.RelinKey(ctx, evk)
    level = n - 1
    # n = 4 and one ciphertext: the least scratch holds no expanded mod-up
    nbytes = (6 * n + 2) * N * 8 * count if minimum else ctx.rotate_scratch_bytes(level, count)
    d = dev(ct)
    out = empty(count, 2, n, N)
    he.rotate(out, d, count, g, key, ctx, level, empty(nbytes // 8))
    got = host(out)
    for c in {0, count - 1}:
        assert np.array_equal(got[c], oracle.rotate(ct[c], g, evk, data, P, level)), c
    he.rotate(d, d, count, g, key, ctx, level, empty(nbytes // 8))
    assert np.array_equal(host(d), got)
