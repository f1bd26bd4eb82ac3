"""The short path of the CRT lift (a coefficient below q_0 / 2 is its centred
residue mod q_0 when every other residue agrees) at its limits, bit-exact
against the oracle's lift: magnitudes around q_0 / 2, and values that agree
with the short path's candidate on all limbs but one."""
import math

import numpy as np
import pytest

from oracle import ckks
from paper_2109_14704_gb300 import he

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.gpu_util import dev, host  # noqa: E402


@pytest.mark.parametrize("bits", [[60], [40, 60], [60, 50, 50, 50], [31] * 5, [60] + [50] * 18])
def test_small_lift_edges(bits):
    N = 1024
    data, P = he.chain_primes(N, bits, 60 if bits[0] < 60 else 59)
    Q, q0 = math.prod(data), data[0]
    h = (Q - 1) // 2
    vals = [0, 1, 2, 1 << 53, (1 << 53) + 1, (1 << 53) + 3, (1 << 54) + 2, (1 << 54) + 6, q0 - 1, q0, q0 + 1]
    vals += [(q0 - 1) // 2 + d for d in range(-3, 4)]
    for i, q in enumerate(data):            # agrees with a small value on every limb but q
        vals += [s + (Q // q) * k for s in (0, 5, -7) for k in (1, q // 2, q - 1)]
    vals = [v for x in vals for v in (x, -x)]
    vals = [(v + h) % Q - h for v in vals]
    vals += [0] * (-len(vals) % N)
    count = len(vals) // N
    res = np.array([[v % q for v in vals] for q in data], dtype=np.uint64)
    coeffs = np.ascontiguousarray(res.reshape(len(data), count, N).transpose(1, 0, 2))
    ctx = he.Context(N, data, P)
    out = torch.empty((count, N), dtype=torch.float64, device="cuda")
    he.Encoder(ctx).crt_compose(out, dev(coeffs), count, len(data) - 1)
    want = np.array([float(v) for v in ckks.crt_centered(res, data)])
    got = out.cpu().numpy().reshape(-1)
    assert np.array_equal(got, want) and not np.signbit(got[got == 0]).any()


def test_decode_leaves_its_input():
    N = 4096
    data, P = he.chain_primes(N, [60, 50], 60)
    ctx = he.Context(N, data, P)
    enc = he.Encoder(ctx)
    z = torch.randn((3, N // 2), dtype=torch.complex128, device="cuda")
    pt = torch.empty((3, 2, N), dtype=torch.int64, device="cuda")
    sc = torch.empty(enc.decode_scratch_bytes(1, 3) // 8, dtype=torch.int64, device="cuda")
    enc.encode(pt, z, 3, 2.0 ** 40, 1, sc)
    before, back = host(pt).copy(), torch.empty_like(z)
    enc.decode(back, pt, 3, 2.0 ** 40, 1, sc)
    assert np.array_equal(host(pt), before) and float((back - z).abs().max()) < 1e-9
