"""The key multiply-accumulate at the ends of its range: the longest chain (32
digits), the smallest and largest primes, every word at its largest, in the
per-tile form (one ciphertext) and the tiled one (8 and 9), bit-exact against
the oracle."""
import numpy as np
import pytest

import oracle
from paper_2109_14704_gb300 import he
from paper_2109_14704_gb300.synth import Rng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.gpu_util import dev, empty, host  # noqa: E402


def _largest(moduli, N, *lead):
    out = np.empty((*lead, len(moduli), N), dtype=np.uint64)
    for i, q in enumerate(moduli):
        out[..., i, :] = q - 1
    return out


@pytest.mark.parametrize("count", [1, 8, 9])
@pytest.mark.parametrize("N,n,bits,level,fill", [(1024, 32, 60, 31, "largest"), (1024, 32, 60, 31, "random"),
                                                 (1024, 6, 31, 5, "largest"), (2048, 2, 40, 1, "random"),
                                                 (1024, 9, 50, 7, "random")])
def test_key_sums(N, n, bits, level, fill, count):
    data, P = he.chain_primes(N, [bits] * n, 60 if bits < 60 else 59)
    r = Rng(N + n + bits)
    if fill == "largest":
        evk = _largest(data + [P], N, n, 2)
    else:
        evk = np.stack([np.stack([r.uniform_limbs(data + [P], N) for _ in range(2)]) for _ in range(n)])
    qs = data[:level + 1]
    ca, cb = _largest(qs, N, count, 2), _largest(qs, N, count, 2)
    if fill == "random":
        for x in (ca, cb):
            for c in range(count):
                x[c] = np.stack([r.uniform_limbs(qs, N) for _ in range(2)])
    else:
        ca[:, :, :, ::3] = 0      # the digits are not all constants
        cb[:, 1, :, 1::7] = 1
    ctx = he.Context(N, data, P)
    key = he.RelinKey(ctx, evk)
    out = empty(count, 2, level, N)
    he.mul_relin_rescale(out, dev(ca), dev(cb), count, key, ctx, level,
                         empty(ctx.mrr_scratch_bytes(level, count) // 8))
    got = host(out)
    want = oracle.mul_relin_rescale(ca[0], cb[0], evk, data, P, level)
    assert np.array_equal(got[0], want)
    for c in {1, count - 1} - {0}:
        if c < count:
            assert np.array_equal(got[c], oracle.mul_relin_rescale(ca[c], cb[c], evk, data, P, level)), c
    # the fused mod-up (minimum scratch) takes the key's other form
    fused = empty(1, 2, level, N)
    he.mul_relin_rescale(fused, dev(ca[:1]), dev(cb[:1]), 1, key, ctx, level,
                         empty(ctx.mrr_scratch_bytes(level, 1, 0) // 8))
    assert np.array_equal(host(fused)[0], want)


def test_key_memory():
    """A key's device copy holds the bytes the ledgers count for it."""
    N, n = 32768, 8
    data, P = he.chain_primes(N, [60] + [50] * (n - 1), 60)
    ctx = he.Context(N, data, P)
    evk = _largest(data + [P], N, n, 2)
    he.RelinKey(ctx, evk).close()                   # the kernels' own memory is in place
    free = torch.cuda.mem_get_info()[0]
    key = he.RelinKey(ctx, evk)
    held = free - torch.cuda.mem_get_info()[0]
    assert he.KEY_BYTES_PER_WORD == 16
    assert evk.size * 16 <= held <= evk.size * 16 + (8 << 20), held      # two allocations, 2 MB pages
    key.close()
