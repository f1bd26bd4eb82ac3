"""The tensor kernel of the encrypted matrix product at the edges of its
output blocks (single rows and columns, odd sizes), at the edge of its sums (32
and 33 terms, largest words), and for the smallest and largest primes."""
import numpy as np
import pytest

import oracle
from paper_2109_14704_gb300 import he
from paper_2109_14704_gb300.synth import Rng

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests.gpu_util import dev, empty, host  # noqa: E402


@pytest.mark.parametrize("m,k,n", [(1, 1, 1), (1, 3, 4), (5, 2, 1), (3, 33, 5), (2, 32, 2), (2, 65, 3)])
@pytest.mark.parametrize("bits,fill", [([60, 60], "largest"), ([31, 31, 31], "largest"), ([60, 40, 31], "random")])
def test_matmul_tensor_shapes(m, k, n, bits, fill):
    N = 1024
    data, P = he.chain_primes(N, bits, 50)
    level = len(data) - 1
    r = Rng(m * 100 + k * 10 + n)
    A = np.empty((m, k, 2, level + 1, N), dtype=np.uint64)
    B = np.empty((k, n, 2, level + 1, N), dtype=np.uint64)
    for X in (A, B):
        for i, q in enumerate(data):
            X[..., i, :] = q - 1 if fill == "largest" else r.uniform_mod(q, X[..., i, :].size).reshape(X[..., i, :].shape)
    if fill == "largest":
        A[..., ::5], B[..., ::7] = 0, 1
    ctx = he.Context(N, data, P)
    out = empty(m, n, 3, level + 1, N)
    he.ct_matmul_tensor(out, dev(A), dev(B), m, k, n, ctx, level)
    got = host(out)
    q = np.array(data, dtype=np.uint64)[None, :, None]
    for i in {0, m - 1}:
        for j in {0, n - 1}:
            want = np.zeros((3, level + 1, N), dtype=np.uint64)
            for l in range(k):
                want = (want + oracle.tensor(A[i, l], B[l, j], data)) % q      # below 2^61: no wrap
            assert np.array_equal(got[i, j], want), (i, j)
