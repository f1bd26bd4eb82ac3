"""Performance cases of the library: what a CKKS program has it do, through
its public entry points (paper_2109_14704_gb300.he), from one small
polynomial to batches that fill the GPU, with odd and ragged sizes.

A case is a dict of plain values; `kind` names the call, the rest its sizes:

  ntt      forward or inverse NTT of `count` polynomials of `limbs` limbs
  plan     one plan of polynomials of mixed degrees and limb counts
  product  negacyclic products of coefficient-domain polynomials
  mrr      Mul + relinearization + rescale of `count` ciphertext pairs
  multi    Mul + relinearization + rescale of jobs of different degrees
  rotate   rotation of `count` ciphertexts
  matmul   encrypted C += A B on matrices of ciphertexts
  codec    encode messages, decode the plaintexts
  encrypt  public-key encryption, randomness drawn on the device

All but `codec` are exact integer arithmetic on residues. `exact` computes
every kind again from its definition in plain torch.
"""
from __future__ import annotations

import random

import numpy as np
import torch

from paper_2109_14704_gb300 import he

DEGREES = (4096, 8192, 16384, 32768)
SCALE = 2.0 ** 40


def listed():
    return [
        # one polynomial under two 60-bit primes: the plain transform call of
        # an interactive program, where the launch is the cost
        dict(name="ntt_fwd_n4096_l2_x1", kind="ntt", N=4096, limbs=2, bits60=2, count=1, inverse=False),
        # a working set of ciphertexts brought back to coefficients
        dict(name="ntt_inv_n16384_l7_x37", kind="ntt", N=16384, limbs=7, bits60=1, count=37, inverse=True),
        # the paper's batched transform: 1024 instances of 8 limbs at 32K
        dict(name="ntt_fwd_n32768_l8_x1024", kind="ntt", N=32768, limbs=8, bits60=4, count=1024, inverse=False),
        # a server's uneven batch: polynomials of every degree and limb count
        dict(name="plan_inv_512", kind="plan", polys=512, max_limbs=16, inverse=True, mix=3),
        # plaintext ring products of a few polynomials
        dict(name="product_n8192_l3_x9", kind="product", N=8192, limbs=3, bits60=1, count=9),
        # one ciphertext product as an interactive evaluation makes it
        dict(name="mrr_n16384_n7_x1", kind="mrr", N=16384, data=7, bits=50, level=6, count=1),
        # the batched ciphertext product (seven 50/60-bit limbs, 64 pairs)
        dict(name="mrr_n16384_n7_x64", kind="mrr", N=16384, data=7, bits=50, level=6, count=64),
        # a serving batch: jobs of three degrees, chains of 17 primes, levels 2 .. 16
        dict(name="multi_16_jobs", kind="multi", jobs=16, data=17, min_log=13, max_log=15, max_level=16,
             max_count=2, mix=5),
        # rotations of the paper's routine set: 32K, 8 limbs, 16 ciphertexts
        dict(name="rotate_n32768_n8_x16", kind="rotate", N=32768, data=8, bits=50, level=7, count=16, steps=1),
        # the paper's encrypted matrix product 10 x 9 x 8 at 8K, 60/40/40 primes
        dict(name="matmul_n8192_10x9x8", kind="matmul", N=8192, data=3, bits=40, level=2, m=10, k=9, n=8),
        # client side: messages to plaintexts and back
        dict(name="codec_n32768_n8_x64", kind="codec", N=32768, data=8, bits=50, level=7, count=64),
        # client side: encryption of a handful of plaintexts
        dict(name="encrypt_n16384_n7_x5", kind="encrypt", N=16384, data=7, bits=50, level=6, count=5),
    ]


def draw(rng):
    largest = [work(c) for c in listed()]
    cap_bytes, cap_flops = max(w["bytes"] for w in largest), max(w["flops"] for w in largest)
    while True:
        case = _draw_any(rng)
        w = work(case)
        # the transforms reach the highest rate; the rest takes up to twice as long an operation
        scale = 1 if case["kind"] in ("ntt", "plan") else 2
        if scale * w["bytes"] <= cap_bytes and scale * w["flops"] <= cap_flops:
            return case


def _log_uniform(rng, lo, hi):
    return min(hi, int(lo * ((hi + 1) / lo) ** rng.random()))


def _draw_any(rng):
    kind = rng.choice(["ntt", "ntt", "plan", "product", "mrr", "mrr", "multi", "rotate", "matmul", "codec",
                       "encrypt"])
    N = rng.choice(DEGREES)
    if kind in ("ntt", "product"):
        N = 1 << rng.randint(10, 16)
        limbs = rng.randint(1, 12)
        return dict(kind=kind, N=N, limbs=limbs, bits60=rng.randint(0, limbs),
                    count=_log_uniform(rng, 1, 1024 if kind == "ntt" else 128), inverse=rng.random() < 0.5)
    if kind == "plan":
        return dict(kind=kind, polys=_log_uniform(rng, 3, 512), max_limbs=rng.randint(1, 16),
                    inverse=rng.random() < 0.5, mix=rng.randint(0, 10 ** 6))
    if kind == "multi":
        return dict(kind=kind, jobs=rng.randint(1, 20), data=rng.randint(2, 17), min_log=12, max_log=15,
                    max_level=16, max_count=_log_uniform(rng, 1, 4), mix=rng.randint(0, 10 ** 6))
    if kind == "matmul":
        return dict(kind=kind, N=rng.choice((4096, 8192)), data=3, bits=rng.choice((40, 50)), level=rng.randint(1, 2),
                    m=rng.randint(1, 12), k=rng.randint(1, 12), n=rng.randint(1, 12))
    data = rng.randint(2, 9)
    case = dict(kind=kind, N=N, data=data, bits=rng.choice((40, 50, 55)), level=rng.randint(1, data - 1),
                count=_log_uniform(rng, 1, 64))
    if kind == "rotate":
        case["steps"] = rng.randint(1, 1000)
    return case


# ------------------------------------------------------------- parameters

def _is_prime(q):
    d, r = q - 1, 0
    while d % 2 == 0:
        d, r = d // 2, r + 1
    for a in (2, 3, 5, 7, 11, 13, 17, 19, 23, 29, 31, 37):
        x = pow(a, d, q)
        if x in (1, q - 1):
            continue
        for _ in range(r - 1):
            x = x * x % q
            if x == q - 1:
                break
        else:
            return False
    return True


def _primes(bits, two_n, count, used=()):
    """The `count` largest primes of `bits` bits that are 1 mod two_n and not in `used`."""
    out = []
    q = ((1 << bits) - 2) // two_n * two_n + 1
    while len(out) < count:
        if q not in used and _is_prime(q):
            out.append(q)
        q -= two_n
    return out


def _moduli(case):
    """Moduli of an ntt or product case: bits60 60-bit primes, then 50-bit ones."""
    return _primes(60, 2 * case["N"], case["bits60"]) + _primes(50, 2 * case["N"], case["limbs"] - case["bits60"])


def _chain(N, data, bits):
    """A 60-bit prime, data - 1 primes of `bits` bits, and the 60-bit special prime."""
    first, special = _primes(60, 2 * N, 2)
    return [first] + _primes(bits, 2 * N, data - 1), special


def _plan_pool():
    return _primes(60, 1 << 16, 6) + _primes(55, 1 << 16, 5) + _primes(50, 1 << 16, 5)


def _plan_polys(case):
    """(N, limbs, first prime) of every polynomial of a plan case."""
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["polys"]):
        limbs = r.randint(1, case["max_limbs"])
        out.append((r.choice(DEGREES), limbs, r.randint(0, 16 - limbs)))
    return out


def _multi_jobs(case):
    """(N, level, count) of every job of a multi case."""
    r = random.Random(case["mix"])
    top = min(case["max_level"], case["data"] - 1)
    degrees = range(case["min_log"], case["max_log"] + 1)
    return [(1 << degrees[j % len(degrees)], r.randint(min(2, top), top), r.randint(1, case["max_count"]))
            for j in range(case["jobs"])]


# ----------------------------------------------------------------- inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed):
    g = torch.Generator(device=_device())
    g.manual_seed(seed)
    return g


def _residues(g, moduli, N, *lead):
    """Uniform residues [*lead][len(moduli)][N]: coefficients and ciphertext
    words are (pseudo-)uniform modulo each prime."""
    out = torch.empty((*lead, len(moduli), N), dtype=torch.int64, device=_device())
    for i, q in enumerate(moduli):
        out[..., i, :] = torch.randint(0, q, (*lead, N), dtype=torch.int64, device=_device(), generator=g)
    return out


def _empty(*shape):
    return torch.empty(shape, dtype=torch.int64, device=_device())


def _key(seed, moduli, N):
    """Key words [digit][2][limb][N]; a real key is pseudo-random modulo each prime."""
    r = np.random.default_rng(seed)
    nd = len(moduli) - 1
    evk = np.empty((nd, 2, nd + 1, N), dtype=np.uint64)
    for t, q in enumerate(moduli):
        evk[:, :, t, :] = r.integers(0, q, (nd, 2, N), dtype=np.uint64)
    return evk


def _slots(g, count, n):
    """Message slots with real and imaginary parts uniform in [-1, 1)."""
    return torch.complex(*(2 * torch.rand((count, n), dtype=torch.float64, device=_device(), generator=g) - 1
                           for _ in range(2)))


def _inputs(case, seed):
    """The seeded data of a case, without any handle of the library."""
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("ntt", "product"):
        qs, N = _moduli(case), case["N"]
        d = dict(moduli=qs, a=_residues(g, qs, N, case["count"]))
        if kind == "product":
            d["b"] = _residues(g, qs, N, case["count"])
        return d
    if kind == "plan":
        # the polynomials lie back to back in one slab, as a server holds them
        pool, polys = _plan_pool(), _plan_polys(case)
        slab = _empty(sum(N * n for N, n, _ in polys))
        views = [v.view(n, N) for v, (N, n, _) in zip(slab.split([N * n for N, n, _ in polys]), polys)]
        for v, (N, n, f) in zip(views, polys):
            v.copy_(_residues(g, pool[f:f + n], N))
        return dict(pool=pool, slab=slab, polys=views)
    if kind == "multi":
        jobs = _multi_jobs(case)
        degrees = sorted({N for N, _, _ in jobs})
        chains = {N: _chain(N, case["data"], 50) for N in degrees}
        evks = {N: _key([seed, N], chains[N][0] + [chains[N][1]], N) for N in degrees}
        cts = [tuple(_residues(g, chains[N][0][:level + 1], N, count, 2) for _ in range(2))
               for N, level, count in jobs]
        return dict(chains=chains, evks=evks, cts=cts)
    N, level = case["N"], case["level"]
    data, special = _chain(N, case["data"], case["bits"])
    qs = data[:level + 1]
    d = dict(data=data, special=special)
    if kind == "codec":
        d["z"] = _slots(g, case["count"], N // 2)
        return d
    if kind == "encrypt":
        d.update(pt=_residues(g, qs, N, case["count"]), pk=_residues(g, data, N, 2),
                 draw_seed=random.Random(seed).getrandbits(64))
        return d
    d["evk"] = _key(seed, data + [special], N)
    if kind == "matmul":
        m, k, n = case["m"], case["k"], case["n"]
        d.update(a=_residues(g, qs, N, m * k, 2), b=_residues(g, qs, N, k * n, 2),
                 c=_residues(g, qs[:-1], N, m * n, 2))
    else:
        d["a"] = _residues(g, qs, N, case["count"], 2)
        if kind == "mrr":
            d["b"] = _residues(g, qs, N, case["count"], 2)
    return d


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind in ("ntt", "product"):
        s["tables"] = he.NttTables(case["N"], s["moduli"])
        if kind == "product":
            s["out"] = torch.empty_like(s["a"])
        return s
    if kind == "plan":
        polys = _plan_polys(case)
        tables = {N: he.NttTables(N, s["pool"]) for N in sorted({p[0] for p in polys})}
        s["plan"] = he.NttPlan([(d, tables[N], N, n, f) for d, (N, n, f) in zip(s["polys"], polys)])
        return s
    if kind == "multi":
        ctx = {N: he.Context(N, *chain) for N, chain in s["chains"].items()}
        key = {N: he.RelinKey(ctx[N], evk) for N, evk in s.pop("evks").items()}
        s["jobs"] = [(_empty(count, 2, level, N), a, b, count, level, key[N], ctx[N])
                     for (a, b), (N, level, count) in zip(s["cts"], _multi_jobs(case))]
        s["scratch"] = _empty(he.mul_relin_rescale_multi_scratch_bytes([j[3:] for j in s["jobs"]]) // 8)
        return s
    N, level = case["N"], case["level"]
    ctx = s["ctx"] = he.Context(N, s["data"], s["special"])
    if kind == "codec":
        s["encoder"] = he.Encoder(ctx)
        s["pt"] = _empty(case["count"], level + 1, N)
        s["out"] = torch.empty_like(s["z"])
        nbytes = max(s["encoder"].encode_scratch_bytes(case["count"]),
                     s["encoder"].decode_scratch_bytes(level, case["count"]))
    elif kind == "encrypt":
        s["out"] = _empty(case["count"], 2, level + 1, N)
        nbytes = ctx.encrypt_scratch_bytes(level, case["count"])
    else:
        s["key"] = he.RelinKey(ctx, s.pop("evk"))
        if kind == "rotate":
            s["out"] = torch.empty_like(s["a"])
            nbytes = ctx.rotate_scratch_bytes(level, case["count"])
        elif kind == "mrr":
            s["out"] = _empty(case["count"], 2, level, N)
            nbytes = ctx.mrr_scratch_bytes(level, case["count"])
        else:
            mn = case["m"] * case["n"]
            s["t"], s["r"] = _empty(mn, 3, level + 1, N), _empty(mn, 2, level, N)
            nbytes = ctx.mrr_scratch_bytes(level, mn)
    s["scratch"] = _empty(nbytes // 8)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "ntt":
        f = he.ntt_inv if case["inverse"] else he.ntt_fwd
        f(s["a"], case["N"], case["limbs"], case["count"], s["tables"])
        return s["a"]
    if kind == "plan":
        s["plan"].inv() if case["inverse"] else s["plan"].fwd()
        return s["slab"]
    if kind == "product":
        he.negacyclic_mul(s["out"], s["a"], s["b"], case["N"], case["limbs"], case["count"], s["tables"])
        return s["out"]
    if kind == "multi":
        he.mul_relin_rescale_multi(s["jobs"], s["scratch"])
        return [j[0] for j in s["jobs"]]
    level, ctx, scratch = case["level"], s["ctx"], s["scratch"]
    if kind == "mrr":
        he.mul_relin_rescale(s["out"], s["a"], s["b"], case["count"], s["key"], ctx, level, scratch)
        return s["out"]
    if kind == "rotate":
        g = pow(5, case["steps"], 2 * case["N"])
        he.rotate(s["out"], s["a"], case["count"], g, s["key"], ctx, level, scratch)
        return s["out"]
    if kind == "matmul":
        m, k, n = case["m"], case["k"], case["n"]
        he.ct_matmul_tensor(s["t"], s["a"], s["b"], m, k, n, ctx, level)
        he.relin_rescale(s["r"], s["t"], m * n, s["key"], ctx, level, scratch)
        he.ct_add(s["c"], s["c"], s["r"], m * n, 2, ctx, level - 1)
        return s["c"]
    if kind == "codec":
        s["encoder"].encode(s["pt"], s["z"], case["count"], SCALE, level, scratch)
        s["encoder"].decode(s["out"], s["pt"], case["count"], SCALE, level, scratch)
        return s["out"]
    he.encrypt_seeded(s["out"], s["pt"], s["pk"], s["draw_seed"], case["count"], ctx, level, scratch)
    return s["out"]


# -------------------------------------------------- least work, tolerances

def work(case):
    """Bytes: every input read once, every output written once (8 bytes a
    word; a key's words once). Flops: 64-bit word operations, three (product,
    sum, difference) to a butterfly, two (product, sum) to a multiply-add."""
    kind = case["kind"]

    def transforms(N, count):
        return 3 * (N // 2) * (N.bit_length() - 1) * count

    def key_switch(N, data, n, count, rescale):
        # per ciphertext: n digits out, n^2 digits in, 2 accumulators out, 2 n
        # lifts in, and for a rescale 2 out and 2 (n - 1) in
        t = n + n * n + 2 + 2 * n + (2 * n if rescale else 0)
        macs = 2 * n * (n + 1) * N
        return 16 * n * (n + 1) * N, count * (transforms(N, t) + 2 * macs)

    if kind in ("ntt", "product"):
        limbs, N = case["limbs"] * case["count"], case["N"]
        if kind == "ntt":
            return dict(bytes=16 * limbs * N, flops=transforms(N, limbs))
        return dict(bytes=24 * limbs * N, flops=transforms(N, 3 * limbs) + limbs * N)
    if kind == "plan":
        polys = _plan_polys(case)
        return dict(bytes=sum(16 * N * n for N, n, _ in polys), flops=sum(transforms(N, n) for N, n, _ in polys))
    if kind == "multi":
        nbytes = flops = 0
        keys = {}
        for N, level, count in _multi_jobs(case):
            n = level + 1
            k, f = key_switch(N, case["data"], n, count, True)
            keys[N] = max(keys.get(N, 0), k)
            nbytes += 8 * N * count * (4 * n + 2 * level)
            flops += f + 7 * n * N * count
        return dict(bytes=nbytes + sum(keys.values()), flops=flops)
    N, n = case["N"], case["level"] + 1
    if kind == "codec":
        c, log = case["count"], N.bit_length() - 2
        # two complex transforms of N / 2 points, two NTTs of every limb
        return dict(bytes=c * N * (8 + 8 + 16 * n), flops=c * (2 * 5 * (N // 2) * log + transforms(N, 2 * n)))
    if kind == "encrypt":
        c = case["count"]
        return dict(bytes=8 * N * n * (3 * c + 2), flops=c * (transforms(N, 3 * n) + 4 * n * N))
    if kind == "matmul":
        m, k, l = case["m"], case["k"], case["n"]
        kb, kf = key_switch(N, case["data"], n, m * l, True)
        return dict(bytes=8 * N * (2 * n * (m * k + k * l) + 4 * (n - 1) * m * l) + kb,
                    flops=8 * m * k * l * n * N + kf + 2 * (n - 1) * N * m * l)
    c = case["count"]
    kb, kf = key_switch(N, case["data"], n, c, kind == "mrr")
    if kind == "mrr":
        return dict(bytes=8 * N * c * (4 * n + 2 * (n - 1)) + kb, flops=kf + 7 * n * N * c)
    return dict(bytes=8 * N * c * 4 * n + kb, flops=kf + n * N * c)


def tolerance(case):
    if case["kind"] == "codec":
        # slots after rounding at scale 2^40: a transform in another order
        # rounds a few coefficients in a million to the other neighbour, and
        # one such step moves every slot of its message by 2^-40, 1.1e-12 of
        # the slots' norm (measured: 3.7e-13 over 64 messages at N = 32768)
        return {"rel": 4e-12}
    return "exact"


# ---------------------------------------------------- definition in 64 bits
#
# Residues below 2^60 as int64. A product a c with c <= 2^30 has a quotient
# below 2^30, which a double estimate gives to within one, and its remainder
# comes from wrapping arithmetic; a full product is made of three of those.

def _mul_small(a, c, q):
    quo = (a.double() * c * (1.0 / q)).floor().to(torch.int64)
    r = a * c - quo * q
    r = torch.where(r < 0, r + q, r)
    return torch.where(r >= q, r - q, r)


def _mul(a, b, q):
    if isinstance(b, int):
        b = torch.tensor(b, dtype=torch.int64, device=a.device)
    hi, lo = b >> 30, b & ((1 << 30) - 1)
    t = _mul_small(_mul_small(a, hi, q), 1 << 30, q)
    return _add(t, _mul_small(a, lo, q), q)


def _add(a, b, q):
    r = a + b
    return torch.where(r >= q, r - q, r)


def _sub(a, b, q):
    r = a - b
    return torch.where(r < 0, r + q, r)


def _powers(w, n, q):
    """1, w, .., w^(n-1) mod q (n a power of two)."""
    p = torch.ones(1, dtype=torch.int64, device=_device())
    while p.numel() < n:
        p = torch.cat([p, _mul(p, pow(w, p.numel(), q), q)])
    return p


def _bit_reverse(n):
    r = torch.zeros(1, dtype=torch.int64, device=_device())
    while r.numel() < n:
        r = torch.cat([2 * r, 2 * r + 1])
    return r


_psi_cache: dict = {}


def _psi(q, N):
    """The smallest primitive 2N-th root of unity mod q."""
    if (q, N) not in _psi_cache:
        g = next(g for g in range(2, 10 ** 4) if pow(g, (q - 1) // 2, q) == q - 1)
        c = pow(g, (q - 1) // (2 * N), q)
        _psi_cache[q, N] = int(_mul(_powers(c * c % q, N, q), c, q).min())
    return _psi_cache[q, N]


def _fwd(x, q):
    """Forward NTT of x [..., N], bit-reversed evaluation order."""
    N = x.shape[-1]
    w = _powers(_psi(q, N), N, q)[_bit_reverse(N)]
    y = x.reshape(-1, N)
    for s in range(N.bit_length() - 1):
        g = 1 << s
        v = y.view(-1, g, 2, N // (2 * g))
        u, t = v[:, :, 0], _mul(v[:, :, 1], w[g:2 * g].view(1, g, 1), q)
        y = torch.stack([_add(u, t, q), _sub(u, t, q)], dim=2).view(-1, N)
    return y.view(x.shape)


def _inv(x, q):
    """Inverse NTT (with 1/N) of x [..., N]."""
    N = x.shape[-1]
    w = _powers(pow(_psi(q, N), -1, q), N, q)[_bit_reverse(N)]
    y = x.reshape(-1, N)
    for s in reversed(range(N.bit_length() - 1)):
        g = 1 << s
        v = y.view(-1, g, 2, N // (2 * g))
        a, b = v[:, :, 0], v[:, :, 1]
        y = torch.stack([_add(a, b, q), _mul(_sub(a, b, q), w[g:2 * g].view(1, g, 1), q)], dim=2).view(-1, N)
    return _mul(y, pow(N, -1, q), q).view(x.shape)


def _limbs(f, x, moduli):
    return torch.stack([f(x[..., i, :].contiguous(), q) for i, q in enumerate(moduli)], dim=-2)


def _tensor(a, b, moduli):
    """(a0 b0, a0 b1 + a1 b0, a1 b1) of a, b [..., 2, n, N]."""
    def comp(i, q):
        a0, a1, b0, b1 = a[..., 0, i, :], a[..., 1, i, :], b[..., 0, i, :], b[..., 1, i, :]
        return torch.stack([_mul(a0, b0, q), _add(_mul(a0, b1, q), _mul(a1, b0, q), q), _mul(a1, b1, q)], dim=-2)
    return torch.stack([comp(i, q) for i, q in enumerate(moduli)], dim=-2)


def _divide(c, y, m, moduli):
    """(c - r) / m on each limb, r the centred residue mod m of coefficients y."""
    r = torch.where(y > (m - 1) // 2, y - m, y)
    return torch.stack([_mul(_sub(c[..., i, :], _fwd(r % q, q), q), pow(m, -1, q), q)
                        for i, q in enumerate(moduli)], dim=-2)


def _relin(c3, evk, data, special):
    """Key switch of c3 [count, 3, n, N]: digits are the residues of c3[2]
    mod each data prime, the sum is divided by the special prime."""
    n, N = c3.shape[-2], c3.shape[-1]
    digits = [_inv(c3[:, 2, j].contiguous(), data[j]) for j in range(n)]
    key = torch.from_numpy(evk.view(np.int64)).to(c3.device)
    acc = []
    for t in list(range(n)) + [len(data)]:
        q = (data + [special])[t]
        s = [0, 0]
        for j in range(n):
            x = c3[:, 2, j] if j == t else _fwd(digits[j] % q, q)
            for k in range(2):
                p = _mul(x, key[j, k, t].view(1, N), q)
                s[k] = p if j == 0 else _add(s[k], p, q)
        acc.append(torch.stack(s, dim=1))                       # [count, 2, N]
    y = _inv(acc[-1], special)
    down = _divide(torch.stack(acc[:-1], dim=-2), y, special, data[:n])
    return torch.stack([_add(c3[:, :2, i], down[..., i, :], q) for i, q in enumerate(data[:n])], dim=-2)


def _rescale(c, moduli):
    last = c[..., -1, :].contiguous()
    return _divide(c[..., :-1, :], _inv(last, moduli[-1]), moduli[-1], moduli[:-1])


def _splitmix(seed, k):
    """Output k of the SplitMix64 stream `seed` (int64 words, logical shifts)."""
    def word(v):
        v &= (1 << 64) - 1
        return v - (1 << 64) if v >> 63 else v

    def shr(x, b):
        return (x >> b) & ((1 << (64 - b)) - 1)
    z = word(seed) + (k + 1) * word(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * word(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * word(0x94D049BB133111EB)
    return z ^ shr(z, 31)


def _draws(seed, count, N):
    """Ternary masks and centred binomial errors [count][3][N] of an encryption."""
    k = torch.arange(3 * count * N, dtype=torch.int64, device=_device()).view(count, 3, N)
    r = _splitmix(seed, k)
    out = sum((r >> b) & 1 for b in range(20)) - sum((r >> b) & 1 for b in range(20, 40))
    r0 = r[:, 0]
    out[:, 0] = (((r0 >> 32) & 0xFFFFFFFF) + (r0 & 0xFFFFFFFF)) % 3 - 1     # 2^32 = 1 mod 3
    return out


def _codec(z):
    """Slots of the rounded polynomial: slot j is its value at zeta^(5^j)."""
    n = z.shape[-1]
    N = 2 * n
    e = torch.tensor([pow(5, j, 2 * N) for j in range(n)], dtype=torch.int64, device=z.device)
    index = (e - 1) // 4
    a = torch.arange(n, dtype=torch.float64, device=z.device) * (np.pi / N)
    zeta = torch.complex(a.cos(), a.sin())
    x = torch.empty_like(z)
    x[:, index] = z * SCALE
    w = torch.view_as_real(torch.fft.fft(x) / n * zeta.conj()).round()
    y = torch.fft.ifft(torch.view_as_complex(w) * zeta) * n
    return y[:, index] / SCALE


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "ntt":
        return _limbs(_inv if case["inverse"] else _fwd, s["a"], s["moduli"])
    if kind == "product":
        def ring(a, b, q):
            return _inv(_mul(_fwd(a.contiguous(), q), _fwd(b.contiguous(), q), q), q)
        return torch.stack([ring(s["a"][:, i], s["b"][:, i], q) for i, q in enumerate(s["moduli"])], dim=1)
    if kind == "plan":
        f = _inv if case["inverse"] else _fwd
        groups, out = {}, s["polys"]
        for p, (N, n, first) in enumerate(_plan_polys(case)):
            for i in range(n):
                groups.setdefault((N, s["pool"][first + i]), []).append((p, i))
        for (N, q), rows in groups.items():
            y = f(torch.stack([s["polys"][p][i] for p, i in rows]), q)
            for row, (p, i) in zip(y, rows):
                out[p][i] = row
        return s["slab"]
    if kind == "multi":
        out = []
        for (a, b), (N, level, _) in zip(s["cts"], _multi_jobs(case)):
            data, special = s["chains"][N]
            qs = data[:level + 1]
            out.append(_rescale(_relin(_tensor(a, b, qs), s["evks"][N], data, special), qs))
        return out
    data, special, qs = s["data"], s["special"], s["data"][:case["level"] + 1]
    N = case["N"]
    if kind == "mrr":
        return _rescale(_relin(_tensor(s["a"], s["b"], qs), s["evk"], data, special), qs)
    if kind == "rotate":
        g = pow(5, case["steps"], 2 * N)
        brv = _bit_reverse(N)
        x = s["a"][..., brv[((g * (2 * brv + 1)) % (2 * N) - 1) // 2]]
        c3 = torch.stack([x[:, 0], torch.zeros_like(x[:, 0]), x[:, 1]], dim=1)
        return _relin(c3, s["evk"], data, special)
    if kind == "matmul":
        m, k, n = case["m"], case["k"], case["n"]
        a, b = s["a"].unflatten(0, (m, k)), s["b"].unflatten(0, (k, n))
        t = None
        for l in range(k):
            p = _tensor(a[:, l, None].expand(m, n, *a.shape[2:]), b[None, l].expand(m, n, *b.shape[2:]), qs)
            t = p if t is None else torch.stack([_add(t[..., i, :], p[..., i, :], q) for i, q in enumerate(qs)], dim=-2)
        r = _rescale(_relin(t.flatten(0, 1), s["evk"], data, special), qs)
        return torch.stack([_add(s["c"][..., i, :], r[..., i, :], q) for i, q in enumerate(qs[:-1])], dim=-2)
    if kind == "codec":
        return _codec(s["z"])
    noise = _draws(s["draw_seed"], case["count"], N)
    out = []
    for i, q in enumerate(qs):
        v, e0, e1 = (_fwd((noise[:, w] % q).contiguous(), q) for w in range(3))
        c0 = _add(_add(_mul(v, s["pk"][0, i][None], q), s["pt"][:, i], q), e0, q)
        out.append(torch.stack([c0, _add(_mul(v, s["pk"][1, i][None], q), e1, q)], dim=1))
    return torch.stack(out, dim=2)
