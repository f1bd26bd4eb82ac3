"""Launches overlap the end of the kernel ahead of them in the stream: long
chains of dependent calls, with other kernels, copies and fills in between, on
one and on two streams, give what the same chain gives with a synchronisation
after every call."""
import numpy as np
import pytest

from paper_2109_14704_gb300 import he

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _chain(sync, streams, N, limbs, reps, seed):
    qs = he.primes_generate(50, 2 * N, limbs)
    t = he.NttTables(N, qs)
    data, P = he.chain_primes(N, [60, 50], 60)
    ctx = he.Context(N, data, P)
    rng = np.random.default_rng(seed)
    evk = np.stack([rng.integers(0, q, (2, 2, N), dtype=np.uint64) for q in data + [P]], axis=2)
    key = he.RelinKey(ctx, evk)
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randint(0, 1 << 40, (limbs, N), dtype=torch.int64, device="cuda", generator=g)
    y, z = x.clone(), torch.empty_like(x)
    ct = torch.randint(0, 1 << 40, (1, 2, 2, N), dtype=torch.int64, device="cuda", generator=g)
    out = torch.zeros((1, 2, 1, N), dtype=torch.int64, device="cuda")
    sc = torch.empty(ctx.rotate_scratch_bytes(1, 1) // 8 + ctx.mrr_scratch_bytes(1, 1) // 8, dtype=torch.int64,
                     device="cuda")
    torch.cuda.synchronize()
    for i in range(reps):
        s = streams[i % len(streams)]
        if i:
            s.wait_stream(streams[(i - 1) % len(streams)])
        with torch.cuda.stream(s):
            steps = [lambda: he.ntt_fwd(x, N, limbs, 1, t), lambda: he.dyadic_mul(z, x, y, N, limbs, 1, t),
                     lambda: y.copy_(z), lambda: he.ntt_inv(z, N, limbs, 1, t), lambda: he.negacyclic_mul(x, z, y, N, limbs, 1, t),
                     lambda: he.rotate(ct, ct, 1, 5, key, ctx, 1, sc),
                     lambda: he.mul_relin_rescale(out, ct, ct, 1, key, ctx, 1, sc),
                     lambda: sc.fill_(-1), lambda: ct[:, :, :1].bitwise_xor_(out & 1)]
            for f in steps:
                f()
                if sync:
                    torch.cuda.synchronize()
    torch.cuda.synchronize()
    return [v.cpu() for v in (x, y, z, ct, out)]


@pytest.mark.parametrize("N,limbs", [(1024, 1), (4096, 3), (32768, 2)])
def test_dependent_chains(N, limbs):
    want = _chain(True, [torch.cuda.current_stream()], N, limbs, 30, N)
    for streams in ([torch.cuda.Stream()], [torch.cuda.Stream(), torch.cuda.Stream()]):
        got = _chain(False, streams, N, limbs, 30, N)
        assert all(torch.equal(a, b) for a, b in zip(want, got))
