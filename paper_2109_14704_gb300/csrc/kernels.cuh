// kernels.cuh -- the CUDA kernels of the library, as templates over the NTT
// shape (words per CTA, CTAs per cluster). inst_n*.cu instantiate them per
// polynomial degree; launch.h describes the host-side launchers.
#pragma once
#include <stdint.h>

#include "launch.h"
#include "ntt_core.cuh"

namespace he {

// ============================================================ plain NTT ====

// Load of a word the kernel does not write (a kernel ahead in the stream may
// have: see stream_order); volatile, so that it stays behind the wait.
__device__ __forceinline__ u64 rd(const u64 *p)
{
    u64 v;
    asm volatile("ld.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ ulonglong2 rd2(const u64 *p)
{
    ulonglong2 v;
    asm volatile("ld.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
    return v;
}

// Bulk tensor store of the forward transform's output (one warp, 16 words
// a thread: thread l of warp w holds the 16 words of row row0 + 32 w + l of
// the tensor map's view, rows of 128 bytes). The warp's rows of the shared
// block are its own from the last exchange on (each thread read back only
// its own row), so it stages them there: 16-byte chunk c of a row goes to
// chunk c ^ (bits 7..9 of the row's address), the 128-byte swizzle, which
// keeps every group of eight lanes on distinct banks. Then one lane issues
// the 4 KB store and waits until it has read the rows (the block is not
// touched again). Against four 256-bit stores a lane, each warp store
// touching 32 lines, the rows leave through the copy engine: measured 1 %
// off the forward transform at N = 2^15.
__device__ __forceinline__ void tma_store_rows(const u64 (&x)[16], u32 wbase, const CUtensorMap *tm, u32 row)
{
    const u32 lane = threadIdx.x & 31u;
    const u32 ra = wbase + lane * 128u;
    const u32 sw = (ra >> 7) & 7u;
#pragma unroll
    for (int c = 0; c < 8; c++)
        asm volatile("st.shared.v2.u64 [%0], {%1, %2};" ::"r"(ra + ((c ^ sw) << 4)), "l"(x[2 * c]), "l"(x[2 * c + 1])
                     : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // visible to the copy engine
    __syncwarp();
    if (lane == 0) {
        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                     ::"l"(tm), "r"(0), "r"(row), "r"(wbase) : "memory");
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
        asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    }
    __syncwarp();
}

// Forward or inverse transform of one limb stored at `data` (in place; the
// inverse reads its input at `src`, which may be another buffer). The forward
// transform's last round and the inverse transform's first round give each
// thread runs of consecutive words, which move as 32-byte quarters (streaming
// cache hints: every word is read and written once per launch); the cross-CTA
// columns move as single coalesced words. Stores are skipped when !valid (idle
// sub-clusters of the mixed-degree kernel). With a tensor map tm (forward, 16
// words a thread, the limb block's first row row0) the output leaves by bulk
// tensor stores instead, where the warp's rows in shared memory are 1024-byte
// aligned (the swizzle's period).
template <class Sh, bool INV>
__device__ __forceinline__ void ntt_limb(u64 *smem, u32 m, u32 rbase, u64 *data, const ulonglong2 *tw,
                                         const PrimeConst &pc, const u64 *src, bool valid = true,
                                         const CUtensorMap *tm = nullptr, u32 row0 = 0)
{
    u64 x[Sh::E];
    const u32 tid = threadIdx.x;
    if constexpr (!INV) {
        auto ld = [&](int P) -> u64 { return __ldcs(reinterpret_cast<const unsigned long long *>(data + P)); };
        auto nost = [&](u32, u64) {};
        ntt_fwd_block<Sh>(smem, m, rbase, tw, pc, ld, nost, x);
        if constexpr (Sh::E == 16) {
            const u32 wbase = smem_u32(smem) + (tid >> 5) * 4096u;
            if (tm && valid && (wbase & 1023u) == 0) {
                tma_store_rows(x, wbase, tm, row0 + (tid >> 5) * 32u);
                return;
            }
        }
        if (valid) {
#pragma unroll
            for (int e = 0; e < Sh::E; e += 4)
                st4_cs(data + last_pos<Sh>(m, tid, e), x[e], x[e + 1], x[e + 2], x[e + 3]);
        }
    } else {
#pragma unroll
        for (int e = 0; e < Sh::E; e += 4)
            ld4_cs(src + last_pos<Sh>(m, tid, e), x[e], x[e + 1], x[e + 2], x[e + 3]);
        auto nold = [&](u32) -> u64 { return 0; };
        auto st = [&](int P, u64 v) {
            if (valid) __stcs(reinterpret_cast<unsigned long long *>(data + P), (unsigned long long)v);
        };
        ntt_inv_block<Sh, true>(smem, m, rbase, tw, pc, nold, st, x);
    }
}

template <class Sh, bool INV>
__device__ __forceinline__ void resolve_item(const NttLaunch &a, u32 item, u64 *&data, const ulonglong2 *&tw,
                                             const PrimeConst *&pcp)
{
    if (a.jobs) {
        const LimbJob &j = a.jobs[item];
        data = j.data;
        tw = INV ? j.tw_inv : j.tw_fwd;
        pcp = j.pc;
    } else {
        data = a.base + (size_t)item * Sh::N;
        const u32 pr = a.first_prime + item % a.limbs;
        tw = (INV ? a.tw_inv : a.tw_fwd) + (size_t)pr * Sh::N;
        pcp = a.pc + pr;
    }
}

// Ask L2 for this CTA's block (B words at m B) of limb `item` of the batch,
// if it exists: one bulk prefetch issued by one thread, no registers held
// and nothing waited for. Limbs read later by other clusters then come from
// L2 instead of HBM, which hides the first-stage load latency.
template <class Sh>
__device__ __forceinline__ void prefetch_limb_block(const NttLaunch &a, u32 item, u32 m)
{
    if (threadIdx.x != 0 || item >= a.items) return;
    const u64 *p = a.jobs ? a.jobs[item].data : (a.src ? a.src : a.base) + (size_t)item * Sh::N;
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p + (size_t)m * Sh::B), "r"(Sh::B * 8u)
                 : "memory");
}

// One cluster per limb. With a.prefetch = the number of co-resident
// clusters, limb item + a.prefetch is the one a cluster started about one
// limb-time from now will take.
template <int LOG_B, int LOG_C, int LOG_E, bool INV, int OCC = 0>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E, OCC>::MIN_CTAS)
k_ntt(const __grid_constant__ NttLaunch a)   // grid constant: tmap is addressed in place
{
    stream_order();
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    extern __shared__ __align__(1024) u64 smem[];
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    const u32 item = blockIdx.x >> LOG_C;
    if (a.prefetch) prefetch_limb_block<Sh>(a, item + a.prefetch, m);
    u64 *data;
    const ulonglong2 *tw;
    const PrimeConst *pcp;
    resolve_item<Sh, INV>(a, item, data, tw, pcp);
    const PrimeConst pc = *pcp;
    if (!INV && a.tma_store)
        ntt_limb<Sh, INV>(smem, m, 0, data, tw, pc, data, true, &a.tmap,
                          (u32)(((size_t)item * Sh::N + m * Sh::B) >> 4));
    else
        ntt_limb<Sh, INV>(smem, m, 0, data, tw, pc, a.src ? a.src + (size_t)item * Sh::N : data);
}

// Persistent form: a fixed grid of clusters walks the limbs (job list or
// uniform batch).
template <int LOG_B, int LOG_C, int LOG_E, bool INV, int OCC = 0>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E, OCC>::MIN_CTAS)
k_ntt_persistent(NttLaunch a)
{
    stream_order();
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    extern __shared__ __align__(16) u64 smem[];
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    const u32 clusters = gridDim.x >> LOG_C;
    bool first = true;
    for (u32 item = blockIdx.x >> LOG_C; item < a.items; item += clusters) {
        if (!first) ntt_barrier<Sh>();
        first = false;
        if (a.prefetch) prefetch_limb_block<Sh>(a, item + clusters, m);   // this cluster's next limb
        u64 *data;
        const ulonglong2 *tw;
        const PrimeConst *pcp;
        resolve_item<Sh, INV>(a, item, data, tw, pcp);
        const PrimeConst pc = *pcp;
        ntt_limb<Sh, INV>(smem, m, 0, data, tw, pc, a.src ? a.src + (size_t)item * Sh::N : data);
    }
}

// Mixed-degree form: clusters of 8 CTAs of 2^12 words each take units of a
// list (plans launch one cluster per unit; a smaller grid walks the list); a
// unit of degree 2^(12+c) holds up to 8 >> c limbs, each transformed by a
// sub-cluster of 2^c CTAs (cluster ranks rbase .. rbase + 2^c - 1). One
// launch covers every degree from 2^12 to 2^15. Sub-clusters without a limb
// in the last unit of a degree recompute the unit's first limb with stores
// switched off, so that every CTA of the cluster passes the same cluster
// barriers. Not inlined: each shape gets its own register allocation (one
// kernel body holding all four shapes spilled up to 656 bytes at 64
// registers; this way 12-44 bytes, 172 for the smallest inverse).
template <class Sh, bool INV>
__device__ __noinline__ void mixed_unit(u64 *smem, u32 rank, const MixedUnit &un, const LimbJob *jobs)
{
    if constexpr (Sh::LOG_C == 3) {
        // the whole cluster transforms the unit's one limb
        const LimbJob j = jobs[un.first_job];
        const PrimeConst pc = *j.pc;
        ntt_limb<Sh, INV>(smem, rank, 0, j.data, INV ? j.tw_inv : j.tw_fwd, pc, j.data);
    } else if constexpr (Sh::LOG_C == 0) {
        // one CTA per limb and no cluster barrier inside the transform: a
        // CTA without a limb has nothing to do
        if (rank >= un.n_jobs) return;
        const LimbJob j = jobs[un.first_job + rank];
        const PrimeConst pc = *j.pc;
        ntt_limb<Sh, INV>(smem, 0, 0, j.data, INV ? j.tw_inv : j.tw_fwd, pc, j.data);
    } else {
        const u32 sub = rank >> Sh::LOG_C;
        const u32 m = rank & (Sh::C - 1);
        const u32 rbase = sub << Sh::LOG_C;
        const bool valid = sub < un.n_jobs;
        const LimbJob j = jobs[un.first_job + (valid ? sub : 0u)];
        const PrimeConst pc = *j.pc;
        ntt_limb<Sh, INV>(smem, m, rbase, j.data, INV ? j.tw_inv : j.tw_fwd, pc, j.data, valid);
    }
}

template <bool INV>
__global__ void __launch_bounds__(256, 4) k_ntt_mixed(const MixedUnit *units, u32 n_units, const LimbJob *jobs)
{
    stream_order();
    extern __shared__ __align__(16) u64 smem[];
    const u32 rank = cluster_ctarank();
    const u32 clusters = gridDim.x >> 3;
    bool first = true;
    for (u32 ui = blockIdx.x >> 3; ui < n_units; ui += clusters) {
        if (!first) cluster_sync_war();
        first = false;
        const MixedUnit un = units[ui];
        switch (un.log_n) {
        case 12: mixed_unit<NttShape<12, 0>, INV>(smem, rank, un, jobs); break;
        case 13: mixed_unit<NttShape<12, 1>, INV>(smem, rank, un, jobs); break;
        case 14: mixed_unit<NttShape<12, 2>, INV>(smem, rank, un, jobs); break;
        default: mixed_unit<NttShape<12, 3>, INV>(smem, rank, un, jobs); break;
        }
    }
}

// ============================================================ fused product

// c = a b mod (X^N + 1, q) for one limb per cluster (Sec. II-B: the
// product of two polynomials is the inverse transform of the pointwise
// product of their transforms): the forward transform of a, its values
// parked in a second shared-memory block (each thread its own positions),
// the forward transform of b, the pointwise Barrett product in registers,
// and the inverse transform straight to c. Per word 16 B are read and 8 B
// written, against 72 B for three separate passes.
template <int LOG_B, int LOG_C, int LOG_E>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E>::NEGA_MIN_CTAS)
k_negacyclic(NegaLaunch a)
{
    stream_order();
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    extern __shared__ __align__(16) u64 smem[];
    u64 *park = smem + Sh::B;                    // [E][T]
    const u32 tid = threadIdx.x;
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    const u32 item = blockIdx.x >> LOG_C;
    const u32 pr = item % a.limbs;
    const PrimeConst pc = a.pc[pr];
    const ulonglong2 *twf = a.tw_fwd + (size_t)pr * Sh::N, *twi = a.tw_inv + (size_t)pr * Sh::N;
    const u64 *A = a.a + (size_t)item * Sh::N, *Bp = a.b + (size_t)item * Sh::N;
    u64 *C = a.c + (size_t)item * Sh::N;
    u64 x[Sh::E];
    auto nost = [&](u32, u64) {};
    // one copy of the forward transform run twice (a loop, not unrolled):
    // two inlined copies let the compiler keep the first one's address and
    // twiddle values live into the second, which spills
#pragma unroll 1
    for (int it = 0; it < 2; it++) {
        const u64 *src = it ? Bp : A;
        if (it) ntt_barrier<Sh>();
        auto ld = [&](int P) -> u64 { return __ldcs(reinterpret_cast<const unsigned long long *>(src + P)); };
        ntt_fwd_block<Sh>(smem, m, 0, twf, pc, ld, nost, x);
        if (it == 0) {
#pragma unroll
            for (int e = 0; e < Sh::E; e++) park[e * Sh::T + tid] = x[e];
        } else {
#pragma unroll
            for (int e = 0; e < Sh::E; e++) x[e] = mul_mod(x[e], park[e * Sh::T + tid], pc);
        }
    }
    ntt_barrier<Sh>();
    auto nold = [&](u32) -> u64 { return 0; };
    auto st = [&](int P, u64 v) { __stcs(reinterpret_cast<unsigned long long *>(C + P), (unsigned long long)v); };
    ntt_inv_block<Sh, true>(smem, m, 0, twi, pc, nold, st, x);
}

// Word of an NTT-domain polynomial that X -> X^g brings to index i. Index i
// holds a(psi^(2 brv(i) + 1)) (the order of he_ntt_fwd), so the image
// sigma(a)(psi^(2 brv(i) + 1)) = a(psi^(g (2 brv(i) + 1))) is the input word at
// index brv((g (2 brv(i) + 1) mod 2N - 1) / 2). The low k bits of i are the
// high k bits of brv(i), which only reach the high k bits of the product: an
// aligned run of 2^k words comes from an aligned run of 2^k words.
__device__ __forceinline__ u32 automorph_index(u32 i, u32 log_n, u32 g)
{
    const u32 mask2 = (2u << log_n) - 1, sh = 32 - log_n;
    const u32 t = (g * (2 * (__brev(i) >> sh) + 1)) & mask2;   // mod 2^32 is enough: 2N divides it
    return __brev((t - 1) >> 1) >> sh;
}

// Randomness of encryption drawn on the device (Sec. II-A Encrypt: a
// uniform ternary mask v and Gaussian-like errors e0, e1). Generator:
// SplitMix64 in counter form (Steele, Lea and Flood 2014): output k of the
// stream with key `seed` is mix(seed + (k + 1) * 0x9E3779B97F4A7C15), with
// mix(z): z = (z ^ z >> 30) * 0xBF58476D1CE4E5B9; z = (z ^ z >> 27) *
// 0x94D049BB133111EB; z ^ z >> 31. Draw w (0: v, 1: e0, 2: e1) of message c
// at coefficient i uses output k = (3 c + w) N + i:
//   v  = (r mod 3) - 1                        (bias below 2^-63)
//   e  = popcount(r & (2^20 - 1)) - popcount((r >> 20) & (2^20 - 1)),
// the centred binomial distribution of parameter 20 (variance 10, standard
// deviation 3.16, |e| <= 20): integer-only, so that any implementation
// following this definition reproduces the draws bit for bit.
__device__ __forceinline__ u64 splitmix64_at(u64 seed, u64 k)
{
    u64 z = seed + (k + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

__device__ __forceinline__ int enc_draw(u64 seed, u32 w, u64 c, u64 i, u32 log_n)
{
    const u64 r = splitmix64_at(seed, ((3 * c + w) << log_n) + i);
    if (w == 0) return (int)(r % 3u) - 1;
    return __popcll(r & 0xFFFFFull) - __popcll((r >> 20) & 0xFFFFFull);
}

#ifdef HE_MISC_KERNELS  // defined by the one translation unit that owns them
// ======================================================== naive radix-2 ====
// The baseline of Sec. III-B: one launch per stage, each thread one
// butterfly, data exchanged through global memory, and a final pass that
// reduces the lazy range to [0, p) (forward) -- 2 N log N + 2 N global
// accesses.

__global__ void k_ntt_naive_stage(NttLaunch a, u32 log_n, u32 S, bool inv)
{
    stream_order();
    const u32 N = 1u << log_n;
    const size_t gid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t total = (size_t)a.items * (N / 2);
    if (gid >= total) return;
    const u32 item = (u32)(gid / (N / 2));
    const u32 b = (u32)(gid % (N / 2));
    u64 *data = a.base + (size_t)item * N;
    const u32 pr = a.first_prime + item % a.limbs;
    const PrimeConst pc = a.pc[pr];
    const u32 t = N >> (S + 1);
    const u32 g = b / t;
    const u32 j = 2 * g * t + (b % t);
    u64 x = data[j], y = data[j + t];
    if (!inv) {
        const ulonglong2 w = a.tw_fwd[(size_t)pr * N + (1u << S) + g];
        ct_butterfly(x, y, w.x, w.y, pc);
    } else if (S == 0) {
        gs_last(x, y, pc);
    } else {
        const ulonglong2 w = a.tw_inv[(size_t)pr * N + inv_tw_pos((int)log_n, (int)S, (int)g)];
        gs_butterfly(x, y, w.x, w.y, pc);
    }
    data[j] = x;
    data[j + t] = y;
}

__global__ void k_ntt_naive_final(NttLaunch a, u32 log_n)
{
    stream_order();
    const u32 N = 1u << log_n;
    const size_t gid = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (size_t)a.items * N) return;
    const u32 item = (u32)(gid >> log_n);
    const PrimeConst &pc = a.pc[a.first_prime + item % a.limbs];
    u64 v = a.base[gid];
    a.base[gid] = reduce_from_fwd_range(v, pc);
}

// =========================================================== dyadic ========

// out = a * b mod q for `items` limbs of N words; 2 words per thread.
__global__ void k_dyadic(u64 *out, const u64 *a, const u64 *b, u32 log_n, u32 items, u32 limbs,
                         u32 first_prime, const PrimeConst *pcs)
{
    stream_order();
    const size_t total2 = ((size_t)items << log_n) >> 1;
    for (size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x; g < total2;
         g += (size_t)gridDim.x * blockDim.x) {
        const size_t e = g * 2;
        const u32 item = (u32)(e >> log_n);
        const PrimeConst pc = pcs[first_prime + item % limbs];
        const ulonglong2 va = *reinterpret_cast<const ulonglong2 *>(a + e);
        const ulonglong2 vb = *reinterpret_cast<const ulonglong2 *>(b + e);
        ulonglong2 r;
        r.x = mul_mod(va.x, vb.x, pc);
        r.y = mul_mod(va.y, vb.y, pc);
        *reinterpret_cast<ulonglong2 *>(out + e) = r;
    }
}

// ============================================================ Mul ==========

// out3[c] = (a0 b0, a0 b1 + a1 b0, a1 b1) per limb (Sec. II-A), count pairs.
__global__ void k_tensor(u64 *out3, const u64 *ct_a, const u64 *ct_b, u32 log_n, u32 n, u32 count,
                         const PrimeConst *pcs)
{
    stream_order();
    const size_t per = (size_t)n << log_n;           // words per component
    const size_t total2 = (size_t)count * per / 2;
    for (size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x; g < total2;
         g += (size_t)gridDim.x * blockDim.x) {
        const size_t e = g * 2;
        const size_t c = e / per;
        const size_t off = e - c * per;
        const u32 limb = (u32)(off >> log_n);
        const PrimeConst pc = pcs[limb];
        const u64 *A = ct_a + c * 2 * per + off;
        const u64 *Bp = ct_b + c * 2 * per + off;
        const ulonglong2 a0 = *reinterpret_cast<const ulonglong2 *>(A);
        const ulonglong2 a1 = *reinterpret_cast<const ulonglong2 *>(A + per);
        const ulonglong2 b0 = *reinterpret_cast<const ulonglong2 *>(Bp);
        const ulonglong2 b1 = *reinterpret_cast<const ulonglong2 *>(Bp + per);
        u64 *O = out3 + c * 3 * per + off;
        ulonglong2 d0, d1, d2;
        d0.x = mul_mod(a0.x, b0.x, pc);
        d0.y = mul_mod(a0.y, b0.y, pc);
        d1.x = mad2_mod(a0.x, b1.x, a1.x, b0.x, pc);
        d1.y = mad2_mod(a0.y, b1.y, a1.y, b0.y, pc);
        d2.x = mul_mod(a1.x, b1.x, pc);
        d2.y = mul_mod(a1.y, b1.y, pc);
        *reinterpret_cast<ulonglong2 *>(O) = d0;
        *reinterpret_cast<ulonglong2 *>(O + per) = d1;
        *reinterpret_cast<ulonglong2 *>(O + 2 * per) = d2;
    }
}

// ct_out = ct_a + ct_b mod q per limb, `words` words of ciphertexts with n
// limbs of 2^log_n words (any number of components), two words per thread.
__global__ void k_ct_add(u64 *out, const u64 *a, const u64 *b, u64 words, u32 log_n, u32 n, const PrimeConst *pcs)
{
    stream_order();
    for (u64 g = (u64)blockIdx.x * blockDim.x + threadIdx.x; 2 * g < words; g += (u64)gridDim.x * blockDim.x) {
        const u64 e = 2 * g;
        const PrimeConst pc = pcs[(u32)((e >> log_n) % n)];
        const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(a + e);
        const ulonglong2 y = *reinterpret_cast<const ulonglong2 *>(b + e);
        *reinterpret_cast<ulonglong2 *>(out + e) = make_ulonglong2(add_mod(x.x, y.x, pc.p), add_mod(x.y, y.y, pc.p));
    }
}

// The automorphism X -> X^g (g odd) on NTT-domain polynomials of 2^log_n
// words (any number of them, back to back): a gather within each polynomial,
// the same for every limb (automorph_index).
__global__ void k_ct_automorph(u64 *out, const u64 *in, u64 words, u32 log_n, u32 g)
{
    stream_order();
    const u32 N = 1u << log_n;
    for (u64 e = (u64)blockIdx.x * blockDim.x + threadIdx.x; e < words; e += (u64)gridDim.x * blockDim.x) {
        const u32 i = (u32)e & (N - 1);
        out[e] = rd(in + (e - i) + automorph_index(i, log_n, g));
    }
}

// ============================================ encrypted matrix product ======
// Tensor part of C += A B (Sec. IV-E matMul_mxnxk; Sec. II-A Mul): for each
// limb and position, T[i][j] = sum_l (a0 b0, a0 b1 + a1 b0, a1 b1) over the
// pairs (A[i][l], B[l][j]) mod q. The three sums of an output are 128-bit
// integers (Sum128) over MM_TERMS terms, the middle one as
// sum (a0 + a1)(b0 + b1) - sum a0 b0 - sum a1 b1 (three products a term
// instead of four; (2^61)^2 32 = 2^127), each reduced once (Montgomery, its
// 2^-64 taken off by a Shoup product with 2^64).
//
// A warp owns 32 positions of one limb and a TI x TJ block of outputs, so a
// term's 2 (TI + TJ) words, loaded as coalesced 256-byte rows, serve TI TJ
// outputs; the four warps of a CTA take neighbouring blocks of the same
// positions and find each other's rows in L1. 84 registers of sums at 2 x 2,
// 168 in all, three CTAs an SM. Measured, 10 x 9 x 8 at N = 2^13, 3 limbs: 118
// us with two columns and two positions a thread and compiled 128-bit sums, 75
// now (the products alone fill the multiply pipe for 26 us); 2 x 1 outputs a
// warp 85, 1 x 2 94, 2 x 2 at two or four CTAs an SM 77 and 80; 32 x 32 x 32
// 4.7 -> 2.1 ms.
constexpr u32 MM_TERMS = 32;

template <int TI, int TJ>
__global__ void __launch_bounds__(128, TI * TJ == 4 ? 3 : 4)
k_ct_matmul_tensor(u64 *t, const u64 *a, const u64 *b, u32 m, u32 k, u32 n, u32 log_n, u32 limbs, u64 warps,
                   const PrimeConst *pcs, const LimbConst *lcs)
{
    stream_order();
    const u64 w = (u64)blockIdx.x * 4 + __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);   // uniform over the warp
    if (w >= warps) return;
    const u32 jt = (n + TJ - 1) / TJ, tiles = (m + TI - 1) / TI * jt;
    const u32 tile = (u32)(w % tiles), i0 = tile / jt * TI, j0 = tile % jt * TJ;
    const u64 pos = w / tiles * 32 + (threadIdx.x & 31);    // limb N + position
    const u32 limb = (u32)(pos >> log_n);
    const size_t poly = (size_t)limbs << log_n;             // words per component
    const PrimeConst pc = pcs[limb];
    const u64 R = lcs[limb].R, R_sh = lcs[limb].R_sh;
    // rows and columns beyond the edge repeat the last one; they are not stored
    const u64 *ap[TI], *bp[TJ];
#pragma unroll
    for (int i = 0; i < TI; i++) ap[i] = a + (size_t)min(i0 + i, m - 1) * k * 2 * poly + pos;
#pragma unroll
    for (int j = 0; j < TJ; j++) bp[j] = b + (size_t)min(j0 + j, n - 1) * 2 * poly + pos;
    const size_t bstep = (size_t)n * 2 * poly;
    for (u32 l0 = 0; l0 < k; l0 += MM_TERMS) {
        Sum128 s[TI][TJ][3];
#pragma unroll
        for (int i = 0; i < TI; i++)
#pragma unroll
            for (int j = 0; j < TJ; j++)
#pragma unroll
                for (int c = 0; c < 3; c++) s[i][j][c].clear();
        const u32 l1 = min(k, l0 + MM_TERMS);
        for (u32 l = l0; l < l1; l++) {
            u64 a0[TI], a1[TI], b0[TJ], b1[TJ];
#pragma unroll
            for (int i = 0; i < TI; i++) a0[i] = *ap[i], a1[i] = ap[i][poly], ap[i] += 2 * poly;
#pragma unroll
            for (int j = 0; j < TJ; j++) b0[j] = *bp[j], b1[j] = bp[j][poly], bp[j] += bstep;
#pragma unroll
            for (int i = 0; i < TI; i++)
#pragma unroll
                for (int j = 0; j < TJ; j++) {
                    s[i][j][0].mac(a0[i], b0[j]);
                    s[i][j][2].mac(a1[i], b1[j]);
                }
#pragma unroll
            for (int i = 0; i < TI; i++) a0[i] += a1[i];
#pragma unroll
            for (int j = 0; j < TJ; j++) b0[j] += b1[j];
#pragma unroll
            for (int i = 0; i < TI; i++)
#pragma unroll
                for (int j = 0; j < TJ; j++) s[i][j][1].mac(a0[i], b0[j]);
        }
#pragma unroll
        for (int i = 0; i < TI; i++)
#pragma unroll
            for (int j = 0; j < TJ; j++) {
                if (i0 + i >= m || j0 + j >= n) continue;
                u64 h[3], lo[3];
#pragma unroll
                for (int c = 0; c < 3; c++) s[i][j][c].total(h[c], lo[c]);
#pragma unroll
                for (int c = 0; c < 3; c += 2)
                    asm("sub.cc.u64 %0, %0, %2;\n\tsubc.u64 %1, %1, %3;"
                        : "+l"(lo[1]), "+l"(h[1]) : "l"(lo[c]), "l"(h[c]));
                u64 *tp = t + ((size_t)(i0 + i) * n + j0 + j) * 3 * poly + pos;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    u64 v = mul_shoup(montgomery_reduce(h[c], lo[c], pc), R, R_sh, pc.p);
                    if (l0) v = add_mod(v, tp[c * poly], pc.p);   // the terms before
                    tp[c * poly] = v;
                }
            }
    }
}

// ============================================================ Encrypt ======

// The draws themselves, as signed 8-bit values [count][N] each.
__global__ void k_enc_draws(int8_t *v, int8_t *e0, int8_t *e1, u64 seed, u32 log_n, u32 count)
{
    stream_order();
    const u64 N = 1ull << log_n, total = (u64)count * N;
    for (u64 e = (u64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (u64)gridDim.x * blockDim.x) {
        const u64 c = e >> log_n, i = e & (N - 1);
        v[e] = (int8_t)enc_draw(seed, 0, c, i, log_n);
        e0[e] = (int8_t)enc_draw(seed, 1, c, i, log_n);
        e1[e] = (int8_t)enc_draw(seed, 2, c, i, log_n);
    }
}

// Public-key encryption (Sec. II-A) from the transformed randomness:
// c0 = v pk0 + pt + e0, c1 = v pk1 + e1 (NTT domain, limb by limb).
// noise [count][3][n][N] (v, e0, e1 transformed), pt [count][n][N],
// pk [2][pk_limbs][N], ct [count][2][n][N].
// Two words a thread; rows (a limb of a message) are counted in 32 bits.
__global__ void k_enc_combine(u64 *ct, const u64 *noise, const u64 *pt, const u64 *pk, u32 log_n, u32 n, u32 count,
                              u32 pk_limbs, const PrimeConst *pcs)
{
    stream_order();
    const size_t N = (size_t)1 << log_n, per = (size_t)n << log_n, pairs = (size_t)count * per / 2;
    for (size_t g = (size_t)blockIdx.x * blockDim.x + threadIdx.x; g < pairs; g += (size_t)gridDim.x * blockDim.x) {
        const u32 row = (u32)(g >> (log_n - 1)), c = row / n, l = row - c * n;
        const size_t P = 2 * g & (N - 1), off = ((size_t)l << log_n) + P;
        const PrimeConst &pc = pcs[l];
        auto ld = [](const u64 *q) { return *reinterpret_cast<const ulonglong2 *>(q); };
        const u64 *z = noise + c * 3 * per + off;
        const ulonglong2 v = ld(z), e0 = ld(z + per), e1 = ld(z + 2 * per), m = ld(pt + 2 * g);
        const ulonglong2 k0 = ld(pk + off), k1 = ld(pk + pk_limbs * N + off);
        auto c0 = [&](u64 a, u64 k, u64 t, u64 e) {
            return add_mod(add_mod(mul_mod(a, k, pc), t, pc.p), e, pc.p);
        };
        u64 *out = ct + c * 2 * per + off;
        *reinterpret_cast<ulonglong2 *>(out) = make_ulonglong2(c0(v.x, k0.x, m.x, e0.x), c0(v.y, k0.y, m.y, e0.y));
        *reinterpret_cast<ulonglong2 *>(out + per) =
            make_ulonglong2(add_mod(mul_mod(v.x, k1.x, pc), e1.x, pc.p), add_mod(mul_mod(v.y, k1.y, pc), e1.y, pc.p));
    }
}
#endif  // HE_MISC_KERNELS

// ============================================== key switching and rescale ==
//
// Relin (Sec. II-A) with RNS digits and one special prime P, as four kernels
// over all ciphertexts of a batch:
//   k_ks_digits   INTT_{q_j}(c[2]_j) -> coefficient digits c2_j     (n INTT)
//   k_ks_modup    for each target t in {q_0..q_l, P}:
//                 acc_k[t] = sum_j NTT_t(c2_j mod t) * evk[j][k][t]  (n^2 NTT)
//                 (for t = q_j the NTT-domain c[2]_j is used as is); on P the
//                 accumulators are brought back by INTT_P and kept as the
//                 coefficient-domain residues y_k = [x_k]_P          (2 INTT);
//                 on the data primes the stored accumulator is already
//                 (acc_k P^-1 + d_k) 2^-64, so that the mod-down needs no d_k:
//   k_ks_moddown  out_k[i] = d_k[i] + (acc_k[q_i] - NTT(r_k mod q_i)) P^-1
//                          = (stored acc - NTT(r_k P^-1 2^-64 mod q_i)) 2^64,
//                 r_k the centred lift of y_k                        (2n NTT)
// RS (Sec. II-A): k_rs_lift brings c_k[q_l] to the coefficient domain
// (2 INTT), k_rs combines (c_k[q_i] - NTT(r mod q_i)) q_l^-1 (2(n-1) NTT).
// MulLinRS fuses Mul into the loads and the two divisions into one transform
// per remaining limb (k_mrr_lift, k_mrr_rest).

// Centred residue of y in [0, m) (|r| <= (m-1)/2) reduced mod q:
// y mod q, or y mod q - m mod q when y > (m-1)/2 (any word y).
__device__ __forceinline__ u64 centred_mod(u64 y, u64 half_m, u64 m_mod_q, const PrimeConst &pc)
{
    const u64 r = reduce_word_canon(y, pc);
    return y > half_m ? sub_mod(r, m_mod_q, pc.p) : r;
}

// a - x + 12p: congruent to a - x mod p and positive for a < 2^63 - 12p and
// x < 12p (a lazy forward-transform output, see ntt_fwd_block with CANON =
// false); below 2^64 for a < 4p (the stored accumulators), so it can go
// straight into mul_shoup.
__device__ __forceinline__ u64 lazy_sub(u64 a, u64 x, u64 twelve_p) { return a + twelve_p - x; }

// Epilogue of a lazy forward transform (ntt_fwd_block with CANON = false):
//   r(e) = (src[P] - x[e]) C mod p,  P = last_pos(e),  C' = Shoup(C),
// for every word the thread holds, into x. Positions e .. e + 3 (e = 0 mod
// 4) of the last round are consecutive and 32-byte aligned, so src moves in
// 32-byte quarters, all of them loaded before the caller stores anything
// (src may be the output: with alternating loads and stores each store
// would evict lines the next loads need).
template <class Sh>
__device__ __forceinline__ void sub_scale_run(u64 (&x)[Sh::E], const u64 *src, u64 C, u64 C_sh,
                                              const PrimeConst &pc, u32 m, u32 tid)
{
    const u64 twelve_p = 3 * pc.four_p;
    u64 v[Sh::E];
#pragma unroll
    for (int e = 0; e < Sh::E; e += 4) ld4(src + last_pos<Sh>(m, tid, e), v[e], v[e + 1], v[e + 2], v[e + 3]);
#pragma unroll
    for (int e = 0; e < Sh::E; e++) x[e] = mul_shoup(lazy_sub(v[e], x[e], twelve_p), C, C_sh, pc.p);
}

// x[] to dst at the thread's last-round positions, in 32-byte quarters.
template <class Sh>
__device__ __forceinline__ void store_run(u64 *dst, const u64 (&x)[Sh::E], u32 m, u32 tid)
{
#pragma unroll
    for (int e = 0; e < Sh::E; e += 4) st4(dst + last_pos<Sh>(m, tid, e), x[e], x[e + 1], x[e + 2], x[e + 3]);
}

// Job of a mixed-level batch that owns global item `item` of stage S (the
// last job whose first item is not above it): its buffers and sizes go into
// a, and the item's index within the job is returned.
__device__ __forceinline__ u32 bind_job(EvalArgs &a, const JobTable &t, int S, u32 item)
{
    u32 lo = 0, hi = t.n_jobs - 1;
    while (lo < hi) {
        const u32 mid = (lo + hi + 1) / 2;
        if (t.job[mid].begin[S] <= item) lo = mid;
        else hi = mid - 1;
    }
    const EvalJob &J = t.job[lo];
    a.ct_a = J.ct_a;
    a.ct_b = J.ct_b;
    a.ct3 = nullptr;
    a.galois = 0;
    a.out = J.out;
    a.c2 = J.c2;
    a.accq = J.accq;
    a.plift = J.plift;
    a.lift2 = J.lift2;
    a.mx = J.mx;
    a.evk_mac = J.evk_mac;
    a.ctx = J.ctx;
    a.n = J.n;
    a.count = J.count;
    a.c_first = 0;
    return item - J.begin[S];
}

// The input of a key switch of one ciphertext. d(k, limb, ..., P): component k of
// its three at position P, from the tensor of the two input ciphertexts (fused
// Mul), from a 3-component input, or through the automorphism.
struct DSource {
    const u64 *ct_a, *ct_b, *ct3;  // per-ciphertext bases
    size_t per;                    // n * N words per component
    u32 galois;                    // nonzero: ct3 = (c0, c1), read as (sigma(c0), 0, sigma(c1))
    // the third component, and its word at position P of a limb
    __device__ __forceinline__ const u64 *third() const { return ct3 + (galois ? per : 2 * per); }
    __device__ __forceinline__ u64 d(int k, u32 limb, u32 log_n, u32 P, const PrimeConst &pc) const
    {
        if (galois) {
            if (k == 1) return 0;
            return rd(ct3 + (k ? per : 0) + ((size_t)limb << log_n) + automorph_index(P, log_n, galois));
        }
        const size_t off = ((size_t)limb << log_n) + P;
        if (ct3) return rd(ct3 + k * per + off);
        if (k == 0) return mul_mod(rd(ct_a + off), rd(ct_b + off), pc);
        if (k == 1) return mad2_mod(rd(ct_a + off), rd(ct_b + per + off), rd(ct_a + per + off), rd(ct_b + off), pc);
        return mul_mod(rd(ct_a + per + off), rd(ct_b + per + off), pc);
    }
    // words P, P + 1 (P even) of a limb row `row` of ct3, through sigma if set:
    // the pair comes from a pair, in either order
    __device__ __forceinline__ ulonglong2 pair(const u64 *row, u32 log_n, u32 P) const
    {
        const u32 src = galois ? automorph_index(P, log_n, galois) : P;
        const ulonglong2 v = rd2(row + (src & ~1u));
        return (src & 1u) ? make_ulonglong2(v.y, v.x) : v;
    }
};

// KIND: the input known at compile time (a kernel that tells them apart at run
// time holds the registers of all three), or SRC_ANY.
template <int KIND = SRC_ANY>
__device__ __forceinline__ DSource dsource(const EvalArgs &a, u32 c)
{
    DSource s;
    s.per = (size_t)a.n * a.ctx.N;
    s.galois = (KIND == SRC_ROTATE || KIND == SRC_ANY) ? a.galois : 0;
    s.ct3 = (KIND == SRC_PAIR || !a.ct3) ? nullptr : a.ct3 + (size_t)c * (s.galois ? 2 : 3) * s.per;
    s.ct_a = a.ct_a ? a.ct_a + (size_t)c * 2 * s.per : nullptr;
    s.ct_b = a.ct_b ? a.ct_b + (size_t)c * 2 * s.per : nullptr;
    if (KIND == SRC_THREE || KIND == SRC_ROTATE) __builtin_assume(s.ct3 != nullptr);
    if (KIND == SRC_ROTATE) __builtin_assume(s.galois != 0);
    return s;
}

// Stage bodies of the MulLinRS pipeline for one item, shared by the per-
// degree kernels (one cluster per item: m = cluster rank, rbase = 0, valid)
// and the multi-degree kernels (multi.cu: sub-clusters of 2^LOG_C CTAs at
// cluster ranks rbase .. rbase + 2^LOG_C - 1; a sub-cluster without an item
// of its own recomputes a valid one with every store switched off, so that
// all CTAs of the cluster pass the same cluster barriers).

// Digit INTT: c2[c][j] = INTT_{q_j}(d2[c][j]), item = c n + j.
template <class Sh, int KIND = SRC_PAIR>
__device__ __forceinline__ void ks_digits_body(const EvalArgs &a, u32 item, u32 m, u32 rbase, bool valid)
{
    extern __shared__ __align__(16) u64 smem[];
    const u32 c = item / a.n, j = item % a.n;
    const DSource ds = dsource<KIND>(a, c);
    const PrimeConst pc = ds.ct3 ? a.ctx.pc[j] : a.ctx.pc_lift[j];
    u64 *out = a.c2 + ((size_t)c * a.n + j) * Sh::N;
    const u32 tid = threadIdx.x;
    u64 x[Sh::E];
    // the thread's inverse-input positions (consecutive quarters): the given
    // third component, or a1 b1 as Montgomery products, below 2 q_j and
    // scaled by 2^-64, which the lift constants' last stage takes off
    if (ds.ct3) {
        const u64 *d = ds.third() + (size_t)j * Sh::N;
        if (ds.galois) {
            // four words come from an aligned run of four, in some order
#pragma unroll
            for (int e = 0; e < Sh::E; e += 4) {
                const u32 P = (u32)last_pos<Sh>(m, tid, e);
                const u32 src = automorph_index(P, Sh::LOG_N, ds.galois);
                u64 v[4];
                ld4(d + (src & ~3u), v[0], v[1], v[2], v[3]);
#pragma unroll
                for (u32 i = 0; i < 4; i++) {
                    const u32 o = (i ? automorph_index(P + i, Sh::LOG_N, ds.galois) : src) & 3u;
                    x[e + i] = (o & 2u) ? ((o & 1u) ? v[3] : v[2]) : ((o & 1u) ? v[1] : v[0]);
                }
            }
        } else {
#pragma unroll
            for (int e = 0; e < Sh::E; e += 4)
                ld4(d + last_pos<Sh>(m, tid, e), x[e], x[e + 1], x[e + 2], x[e + 3]);
        }
    } else {
        const size_t off = ds.per + (size_t)j * Sh::N;
#pragma unroll
        for (int e = 0; e < Sh::E; e += 4) {
            const int P = last_pos<Sh>(m, tid, e);
            u64 b[4];
            ld4(ds.ct_a + off + P, x[e], x[e + 1], x[e + 2], x[e + 3]);
            ld4(ds.ct_b + off + P, b[0], b[1], b[2], b[3]);
#pragma unroll
            for (int i = 0; i < 4; i++) x[e + i] = mul_mont(x[e + i], b[i], pc);
        }
    }
    auto nold = [&](u32) -> u64 { return 0; };
    auto st = [&](u32 P, u64 v) {
        if (valid) out[P] = v;
    };
    ntt_inv_block<Sh, true>(smem, m, rbase, a.ctx.tw_inv + (size_t)j * Sh::N, pc, nold, st, x);
}

template <int LOG_B, int LOG_C, int LOG_E, bool JOBS = false>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E>::MIN_CTAS)
k_ks_digits(EvalArgs a0, JobsArg<JOBS> tab)
{
    stream_order();
    EvalArgs a = a0;
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    u32 item = blockIdx.x >> LOG_C;
    if constexpr (JOBS) item = bind_job(a, tab, JS_DIGITS, item);
    ks_digits_body<Sh>(a, item, m, 0, true);
}

// The same for given three-component inputs and for rotations.
template <int LOG_B, int LOG_C, int LOG_E, int KIND>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E>::MIN_CTAS)
k_ks_digits_of(EvalArgs a)
{
    stream_order();
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    ks_digits_body<NttShape<LOG_B, LOG_C, LOG_E>, KIND>(a, blockIdx.x >> LOG_C, m, 0, true);
}

template <int LOG_B, int LOG_C, int LOG_E>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E>::EVAL_MIN_CTAS)
k_ks_modup(EvalArgs a)
{
    stream_order();
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    extern __shared__ __align__(16) u64 smem[];
    u64 *acc = smem + Sh::B;                   // [2][E][T], own positions only
    const u32 tid = threadIdx.x;
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    const u32 item = blockIdx.x >> LOG_C;
    const u32 n = a.n;
    const u32 c = item / (n + 1), t = item % (n + 1);
    const u32 tp = (t == n) ? a.ctx.n_data : t; // prime index of the target
    const PrimeConst pc = a.ctx.pc[tp];
    const DSource ds = dsource(a, c);
    const ulonglong2 *twf = a.ctx.tw_fwd + (size_t)tp * Sh::N;
    u64 x[Sh::E];
    for (u32 j = 0; j < n; j++) {
        if (t == j) {
            // the NTT-domain digit times 2^-64, which its key words take off
            const LimbConst &lc = a.ctx.limb[t];
#pragma unroll
            for (int e = 0; e < Sh::E; e++)
                x[e] = mul_shoup_lazy4_asm(ds.d(2, j, Sh::LOG_N, last_pos<Sh>(m, tid, e), pc), lc.k2, lc.k2_sh, pc.neg_p);
        } else {
            if (j > 0) ntt_barrier<Sh>();
            const u64 *src = a.c2 + ((size_t)c * n + j) * Sh::N;
            auto st = [&](u32, u64) {};
            // The transform takes any input below 8t + 2^32 congruent to the
            // digit: when q_j <= 8t the digit c2_j < q_j goes in as it is.
            if (a.ctx.pc[j].p <= (pc.four_p << 1)) {
                auto ld = [&](u32 P) -> u64 { return rd(src + P); };
                ntt_fwd_block<Sh, false>(smem, m, 0, twf, pc, ld, st, x);
            } else {
                auto ld = [&](u32 P) -> u64 {
                    return reduce_word(rd(src + P), pc);
                };
                ntt_fwd_block<Sh, false>(smem, m, 0, twf, pc, ld, st, x);
            }
        }
        // multiply-accumulate with the key: lazy products in [0, 4p),
        // accumulators kept in [0, 4p). Words and quotients come from two arrays
        // in 256-bit loads (64 products at 2^14, 7 + 1 primes, 1278 us; with
        // 128-bit loads 1467, with interleaved pairs in 128-bit loads 1404)
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const size_t row = (((size_t)j * 2 + k) * (a.ctx.n_data + 1) + tp) * Sh::N;
#pragma unroll
            for (int e = 0; e < Sh::E; e += 4) {
                const size_t at = row + last_pos<Sh>(m, tid, e);
                u64 w[4], w_sh[4];
                ld4_nc(a.evk_mac + at, w[0], w[1], w[2], w[3]);
                ld4_nc(a.evk_sh + at, w_sh[0], w_sh[1], w_sh[2], w_sh[3]);
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const u64 prod = mul_shoup_lazy4_asm(x[e + i], w[i], w_sh[i], pc.neg_p);
                    u64 &slot = acc[(k * Sh::E + e + i) * Sh::T + tid];
                    slot = (j == 0) ? prod : reduce_once(slot + prod, pc.four_p);
                }
            }
        }
    }
    if (t < n) {
        // (acc_k P^-1 + d_k) 2^-64, below 4 q_t (the key words hold P^-1)
        const LimbConst lc = a.ctx.limb[t];
#pragma unroll
        for (int k = 0; k < 2; k++) {
            u64 *dst = a.accq + (((size_t)c * 2 + k) * n + t) * Sh::N;
#pragma unroll
            for (int e = 0; e < Sh::E; e++) {
                const int P = last_pos<Sh>(m, tid, e);
                const u64 s = mul_shoup_lazy4_asm(acc[(k * Sh::E + e) * Sh::T + tid], lc.k2, lc.k2_sh, pc.neg_p);
                const u64 d = mul_shoup_lazy4_asm(ds.d(k, t, Sh::LOG_N, (u32)P, pc), lc.k2, lc.k2_sh, pc.neg_p);
                dst[P] = reduce_once(s + d, pc.four_p);
            }
        }
    } else {
        // special prime: y_k = INTT_P(acc_k), kept in the coefficient domain; the
        // sums are 2^64 acc_k there (the key words' scale)
#pragma unroll 1
        for (int k = 0; k < 2; k++) {
            ntt_barrier<Sh>();
#pragma unroll
            for (int e = 0; e < Sh::E; e++) x[e] = montgomery_reduce(0, acc[(k * Sh::E + e) * Sh::T + tid], pc);
            u64 *dst = a.plift + ((size_t)c * 2 + k) * Sh::N;
            auto st = [&](u32 P, u64 v) { dst[P] = v; };
            auto ld = [&](u32) -> u64 { return 0; };
            ntt_inv_block<Sh, true>(smem, m, 0, a.ctx.tw_inv + (size_t)tp * Sh::N, pc, ld, st, x);
        }
    }
}

// Expanded mod-up, first half: one transform per cluster,
//   X[g][t][j] = NTT_t(c2_j mod t)  for each digit j != t, target t in
//   {q_0..q_l, P}, ciphertext c = c_first + g of the group,
// left in the lazy range [0, 8t + 2^32): the 128-bit key sums (MacSums::digit)
// rely on that bound, not only on 12t, which would overflow them. The same
// transforms as k_ks_modup, but as independent launches of the plain
// transform's size and register budget instead of a sequence inside one
// accumulating cluster; k_ks_mac or k_ks_mac_tiled then accumulates them.
// Clusters of the diagonal (j = t) exit at once: there the digit is already
// in the NTT domain.
// One transform of the expanded mod-up: X[g][t][j] = NTT_t(c2_j mod t),
// j != t, ciphertext c_first + g.
template <class Sh>
__device__ __forceinline__ void ks_expand_body(const EvalArgs &a, u32 g, u32 t, u32 j, u32 m, u32 rbase, bool valid)
{
    extern __shared__ __align__(16) u64 smem[];
    const u32 tid = threadIdx.x;
    const u32 n = a.n;
    const u32 tp = (t == n) ? a.ctx.n_data : t;
    const PrimeConst pc = a.ctx.pc[tp];
    const u64 *src = a.c2 + ((size_t)(a.c_first + g) * n + j) * Sh::N;
    u64 *dst = a.mx + (((size_t)g * (n + 1) + t) * n + j) * Sh::N;
    const ulonglong2 *twf = a.ctx.tw_fwd + (size_t)tp * Sh::N;
    u64 x[Sh::E];
    auto nost = [&](u32, u64) {};
    // any input below 8t congruent to the digit will do: when q_j <= 8t the
    // digit c2_j < q_j goes in as it is, otherwise reduce_word brings it
    // below 4t. One transform for both (the flag is uniform over the
    // item): two instances of the transform in one kernel spilled 132 bytes
    // at 64 registers, one spills 8 (measured 1.8 % off the MulLinRS batch).
    const bool reduce = a.ctx.pc[j].p > (pc.four_p << 1);
    auto ld = [&](int P) -> u64 {
        const u64 v = rd(src + P);
        return reduce ? reduce_word(v, pc) : v;
    };
    ntt_fwd_block<Sh, false>(smem, m, rbase, twf, pc, ld, nost, x);
    if (valid) store_run<Sh>(dst, x, m, tid);
}

template <int LOG_B, int LOG_C, int LOG_E, bool JOBS = false>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E>::MIN_CTAS)
k_ks_expand(EvalArgs a0, JobsArg<JOBS> tab)
{
    stream_order();
    EvalArgs a = a0;
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    u32 item = blockIdx.x >> LOG_C;
    if constexpr (JOBS) item = bind_job(a, tab, JS_EXPAND, item);
    const u32 n = a.n;
    const u32 j = item % n, t = (item / n) % (n + 1), g = item / (n * (n + 1));
    if (j == t) return;   // the whole cluster: there the digit is already in the NTT domain
    ks_expand_body<Sh>(a, g, t, j, m, 0, true);
}

#ifdef HE_MISC_KERNELS
// Expanded mod-up, second half (elementwise): for target t and component k
//   acc_k = sum_j X[g][t][j] * evk[j][k][t]   (j = t: the NTT-domain digit
// d2_t itself). The sums are 128-bit integers (Sum128) reduced once by
// Montgomery's 2^-64, with the factors the division needs folded into the
// uploaded key words: on the data primes P^-1, so that the tensor terms d_k
// (products of two canonical words) join the same sum, giving
// (acc_k P^-1 + d_k) 2^-64 in accq; on the special prime 2^64, giving acc_k in
// plift. The diagonal digit enters as a Montgomery product, whose 2^-64 its
// key words take off. All results in [0, 4 p).
// Bounds: x is brought below 4 p + 2^32 <= 8 p (2^30 <= p < 2^60), so 32
// digits and two tensor products sum to less than 2^128, and the reduced sum
// is below 10 p.

// Words at two neighbouring positions.
struct MacVec {
    u64 v[2];
    __device__ __forceinline__ static MacVec load(const u64 *p)
    {
        const ulonglong2 t = rd2(p);
        return {{t.x, t.y}};
    }
    __device__ __forceinline__ static MacVec key(const u64 *p)   // read-only path: key words
    {
        const ulonglong2 t = __ldg(reinterpret_cast<const ulonglong2 *>(p));
        return {{t.x, t.y}};
    }
    __device__ __forceinline__ static MacVec of(ulonglong2 t) { return {{t.x, t.y}}; }
    __device__ __forceinline__ static MacVec shared(const u64 *p)
    {
        const ulonglong2 t = *reinterpret_cast<const ulonglong2 *>(p);
        return {{t.x, t.y}};
    }
    __device__ __forceinline__ void store(u64 *p) const
    {
        *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(v[0], v[1]);
    }
};

// The sums at positions P, P + 1 of one target for one ciphertext.
struct MacSums {
    using Vec = MacVec;
    Sum128 s[2][2];   // [component][position]

    __device__ __forceinline__ void add(const Vec &x, int k, const Vec &w)
    {
#pragma unroll
        for (int i = 0; i < 2; i++) s[k][i].mac(x.v[i], w.v[i]);
    }
    // a transformed digit: the lazy output below 8 p + 2^32 to below 4 p + 2^32
    __device__ __forceinline__ void digit(Vec x, const Vec &w0, const Vec &w1, const PrimeConst &pc)
    {
#pragma unroll
        for (int i = 0; i < 2; i++)
            if ((u32)(x.v[i] >> 32) >= pc.h4) x.v[i] -= pc.four_p;
        add(x, 0, w0);
        add(x, 1, w1);
    }
    // the tensor terms and the diagonal digit, whose key words are w0, w1
    // (none on the special prime)
    __device__ __forceinline__ void begin(const DSource &ds, u32 t, u32 n, u32 log_n, u32 P, const PrimeConst &pc,
                                          const Vec &w0, const Vec &w1, const LimbConst *limb)
    {
#pragma unroll
        for (int k = 0; k < 2; k++)
#pragma unroll
            for (int i = 0; i < 2; i++) s[k][i].clear();
        if (t == n) return;
        Vec d;
        if (ds.ct3) {
            const LimbConst &lc = limb[t];
            d = Vec::of(ds.pair(ds.third() + ((size_t)t << log_n), log_n, P));
#pragma unroll
            for (int i = 0; i < 2; i++) d.v[i] = mul_shoup_lazy4_asm(d.v[i], lc.k2, lc.k2_sh, pc.neg_p);
        } else {
            const size_t off = ((size_t)t << log_n) + P;
            const Vec a0 = Vec::load(ds.ct_a + off), a1 = Vec::load(ds.ct_a + ds.per + off);
            const Vec b0 = Vec::load(ds.ct_b + off), b1 = Vec::load(ds.ct_b + ds.per + off);
            add(a0, 0, b0);
            add(a0, 1, b1);
            add(a1, 1, b0);
#pragma unroll
            for (int i = 0; i < 2; i++) d.v[i] = mul_mont(a1.v[i], b1.v[i], pc);
        }
        add(d, 0, w0);
        add(d, 1, w1);
    }
    __device__ __forceinline__ void finish(const EvalArgs &a, const DSource &ds, u32 c, u32 t, u32 log_n, u32 P,
                                           const PrimeConst &pc) const
    {
        const u32 n = a.n, N = a.ctx.N;
#pragma unroll
        for (int k = 0; k < 2; k++) {
            Vec o;
#pragma unroll
            for (int i = 0; i < 2; i++) o.v[i] = s[k][i].redc(pc);
            u64 *dst;
            if (t < n) {
                if (ds.ct3 && !(k == 1 && ds.galois)) {
                    const LimbConst &lc = a.ctx.limb[t];
                    const Vec d = Vec::of(ds.pair(ds.ct3 + k * ds.per + ((size_t)t << log_n), log_n, P));
#pragma unroll
                    for (int i = 0; i < 2; i++) o.v[i] += mul_shoup_lazy4_asm(d.v[i], lc.k2, lc.k2_sh, pc.neg_p);
                }
                dst = a.accq + (((size_t)c * 2 + k) * n + t) * N + P;
            } else {
                dst = a.plift + ((size_t)c * 2 + k) * N + P;
            }
#pragma unroll
            for (int i = 0; i < 2; i++) o.v[i] = reduce_once(reduce_once(o.v[i], pc.four_p << 1), pc.four_p);
            o.store(dst);
        }
    }
};

// One tile: MAC_BLOCK positions of one target for one ciphertext of the
// group, two to a thread; the ciphertexts of a group are neighbouring
// tiles, so that they find each other's key words in L2. The next digit's
// words are loaded while the current products run.
constexpr u32 MAC_BLOCK = 512;

template <int KIND>
__device__ __forceinline__ void ks_mac_tile(const EvalArgs &a, u32 groups, u32 tile)
{
    using Vec = MacVec;
    const u32 n = a.n, N = a.ctx.N, nd1 = a.ctx.n_data + 1;
    const u32 log_n = 31 - __clz(N), per = N / MAC_BLOCK;
    const u32 g = tile % groups, r = tile / groups;
    const u32 P = (r % per) * MAC_BLOCK + threadIdx.x * 2, t = r / per;
    const u32 tp = (t == n) ? a.ctx.n_data : t;
    const PrimeConst pc = a.ctx.pc[tp];
    const u32 c = a.c_first + g;
    const DSource ds = dsource<KIND>(a, c);
    const size_t key_k = (size_t)nd1 * N, key_j = 2 * key_k;             // evk [j][k][target][N]
    const u64 *key = a.evk_mac + (size_t)tp * N + P;
    const u64 *mx = a.mx + ((size_t)g * (n + 1) + t) * n * N + P;        // mx [g][target][j][N]
    const u64 *kt = key + (t < n ? t : 0) * key_j;
    MacSums acc;
    acc.begin(ds, t, n, log_n, P, pc, Vec::key(kt), Vec::key(kt + key_k), a.ctx.limb);
    // the digits j != t: n of them on the special prime, n - 1 otherwise
    const u32 terms = t < n ? n - 1 : n;
    u32 j = t == 0 ? 1u : 0u;
    Vec v, w0, w1;
    if (terms) v = Vec::load(mx + (size_t)j * N), w0 = Vec::key(key + j * key_j), w1 = Vec::key(key + j * key_j + key_k);
    for (u32 i = 0; i < terms; i++) {
        const Vec x = v, k0 = w0, k1 = w1;
        if (i + 1 < terms) {
            j += j + 1 == t ? 2u : 1u;
            v = Vec::load(mx + (size_t)j * N), w0 = Vec::key(key + j * key_j), w1 = Vec::key(key + j * key_j + key_k);
        }
        acc.digit(x, k0, k1, pc);
    }
    acc.finish(a, ds, c, t, log_n, P, pc);
}

// Tiles of a uniform group (groups x (n + 1) targets x N / MAC_BLOCK), or
// those of every job of a table back to back (each job one group of all its
// ciphertexts).
template <bool JOBS, int KIND>
__global__ void __launch_bounds__(MAC_BLOCK / 2, 4) k_ks_mac(EvalArgs a0, u32 groups, u32 total, JobsArg<JOBS> tab)
{
    stream_order();
    for (u32 q = blockIdx.x; q < total; q += gridDim.x) {
        if constexpr (JOBS) {
            EvalArgs a = a0;
            const u32 local = bind_job(a, tab, JS_MAC, q);
            ks_mac_tile<KIND>(a, a.count, local);
        } else {
            ks_mac_tile<KIND>(a0, groups, q);
        }
    }
}

// Form for a uniform group of at least 8 ciphertexts: one CTA per (target t,
// tile of MAC_TILE positions, chunk of MAC_CHUNK ciphertexts), a warp per
// ciphertext at a time. The tile's key words for every digit and component
// are staged in shared memory once ([2 j + k][position]) and serve every
// ciphertext of the chunk. Same sums, so the outputs are those of k_ks_mac.
// Bound by the multiply pipe (69 % busy) with HBM at 60 %: at N = 2^14, n = 7,
// 64 ciphertexts (470 MB of digits, 780 MB in all) 257 us with a lazy Shoup
// product per term and a separate d_k P, 183 us with the sums. Four CTAs an SM
// (64 registers): three or five 5 to 6 % slower on the whole batch, one
// position a thread at six 4 % slower, a shared-memory queue of asynchronous
// copies 4 % slower (more instructions; the loads are not what it waits for).
constexpr u32 MAC_TILE = 64, MAC_CHUNK = 32;

template <int KIND>
__global__ void __launch_bounds__(256, 4) k_ks_mac_tiled(EvalArgs a, u32 groups)
{
    stream_order();
    using Vec = MacVec;
    extern __shared__ __align__(16) u64 key_tile[];   // [2 n][MAC_TILE]
    const u32 n = a.n, N = a.ctx.N, nd1 = a.ctx.n_data + 1;
    const u32 tiles = N / MAC_TILE, chunks = (groups + MAC_CHUNK - 1) / MAC_CHUNK;
    const u32 b = blockIdx.x;
    const u32 chunk = b % chunks, tile = (b / chunks) % tiles, t = b / (chunks * tiles);
    const u32 tp = (t == n) ? a.ctx.n_data : t;
    const PrimeConst pc = a.ctx.pc[tp];
    const u32 P0 = tile * MAC_TILE;
    const u32 lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const u32 gend = min(groups, (chunk + 1) * MAC_CHUNK);
    // ask L2 for the digit rows of the warp's first ciphertext, 512 bytes each,
    // while the key tile is staged (900 -> 888 us for the batch of 64; asking
    // for every next ciphertext as well 894, for the tensor rows too 903)
    if (chunk * MAC_CHUNK + warp < gend) {
        const u64 *rows = a.mx + ((size_t)(chunk * MAC_CHUNK + warp) * (n + 1) + t) * n * N + P0;
        for (u32 i = lane; i < 4 * n; i += 32)
            if (i / 4 != t) asm volatile("prefetch.global.L2 [%0];" ::"l"(rows + (size_t)(i / 4) * N + i % 4 * 16));
    }
    for (u32 i = 2 * threadIdx.x; i < n * 2 * MAC_TILE; i += 2 * blockDim.x) {
        const u32 row = i / MAC_TILE, col = i % MAC_TILE;   // row 2 j + k: evk [j][k][target][N]
        MacVec::key(a.evk_mac + ((size_t)row * nd1 + tp) * N + P0 + col).store(key_tile + i);
    }
    __syncthreads();
    const u32 P = P0 + 2 * lane;
    const u32 log_n = 31 - __clz(N);
    const u64 *kl = key_tile + 2 * lane;
    for (u32 g = chunk * MAC_CHUNK + warp; g < gend; g += 8) {
        const u64 *mx = a.mx + ((size_t)g * (n + 1) + t) * n * N + P;   // mx [g][target][j][N]
        const u32 c = a.c_first + g;
        const DSource ds = dsource<KIND>(a, c);
        const u32 terms = t < n ? n - 1 : n, jt = t < n ? t : 0;
        u32 j = t == 0 ? 1u : 0u;
        Vec v;
        if (terms) v = Vec::load(mx + (size_t)j * N);
        MacSums acc;
        acc.begin(ds, t, n, log_n, P, pc, Vec::shared(kl + 2 * jt * MAC_TILE),
                  Vec::shared(kl + (2 * jt + 1) * MAC_TILE), a.ctx.limb);
        for (u32 i = 0; i < terms; i++) {
            const Vec x = v;
            const u64 *w = kl + 2 * j * MAC_TILE;
            if (i + 1 < terms) {
                j += j + 1 == t ? 2u : 1u;
                v = Vec::load(mx + (size_t)j * N);
            }
            acc.digit(x, Vec::shared(w), Vec::shared(w + MAC_TILE), pc);
        }
        acc.finish(a, ds, c, t, log_n, P, pc);
    }
}

// Device words of an uploaded key, [nd][2][nd + 1][N] canonical words in mac:
// replaced by the key sums' words w (scaled as EvalArgs says), with their Shoup
// quotients in sh for the fused mod-up. The quotient floor(w 2^64 / p) comes in
// two steps of 32 bits: with mu = floor(2^(2b+2) / p) and r < p < 2^b, r mu /
// 2^(2b-30) is r 2^32 / p less below one, so its floor is short by at most two.
__device__ __forceinline__ u64 shoup_step(u64 &r, const PrimeConst &c)
{
    u64 hi, lo;
    mul_wide(r, c.mu, hi, lo);
    const u32 s = 2 * c.bits - 30;               // 32 .. 90
    u64 q = s < 64 ? (hi << (64 - s)) | (lo >> s) : hi >> (s - 64);
    r = (r << 32) - q * c.p;                     // below 3 p
    while (r >= c.p) r -= c.p, q++;
    return q;
}

__global__ void k_key_prepare(u64 *mac, u64 *sh, u64 words, u32 log_n, u32 nd, const PrimeConst *pcs,
                              const LimbConst *limb, u64 R_special)
{
    stream_order();
    for (u64 e = (u64)blockIdx.x * blockDim.x + threadIdx.x; e < words; e += (u64)gridDim.x * blockDim.x) {
        const u32 t = (u32)((e >> log_n) % (nd + 1));
        const PrimeConst pc = pcs[t];
        const u32 j = (u32)((e >> log_n) / (2 * (nd + 1)));
        u64 f = R_special;
        if (t < nd) f = j == t ? mul_mod(limb[t].Pinv, limb[t].R, pc) : limb[t].Pinv;
        const u64 w = mul_mod(mac[e], f, pc);
        u64 r = w;
        const u64 qh = shoup_step(r, pc);
        const u64 ql = shoup_step(r, pc);
        mac[e] = w;
        sh[e] = (qh << 32) + ql;
    }
}
#endif  // HE_MISC_KERNELS

// Relin mod-down (no rescale): out[c][k][i] = d_k[i] + (acc - NTT(r)) P^-1,
// at the accumulator's scale: (stored acc - NTT(r P^-1 2^-64)) 2^64, with
// r P^-1 = y P^-1 - 1 where y is above half.
// One transform a limb at the plain transform's register budget (at 126
// registers, two CTAs of 256 an SM, 126 us for 256 limbs of 2^15 words; at 64
// 98 us).
template <int LOG_B, int LOG_C, int LOG_E>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E>::MIN_CTAS)
k_ks_moddown(EvalArgs a)
{
    stream_order();
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    extern __shared__ __align__(16) u64 smem[];
    const u32 tid = threadIdx.x;
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    const u32 item = blockIdx.x >> LOG_C;
    const u32 n = a.n;
    const u32 c = item / (2 * n), k = (item / n) % 2, i = item % n;
    const PrimeConst pc = a.ctx.pc[i];
    const PrimeConst pP = a.ctx.pc[a.ctx.n_data];
    const LimbConst lc = a.ctx.limb[i];
    const u64 half_P = (pP.p - 1) / 2, minus_k2 = pc.p - lc.k2;
    const u64 *y = a.plift + ((size_t)c * 2 + k) * Sh::N;
    u64 x[Sh::E];
    auto ld = [&](u32 P) -> u64 {   // below 5 q_i
        const u64 v = rd(y + P);
        return mul_shoup_lazy4_asm(v, lc.k1, lc.k1_sh, pc.neg_p) + (v > half_P ? minus_k2 : 0);
    };
    auto st = [&](u32, u64) {};
    ntt_fwd_block<Sh, false>(smem, m, 0, a.ctx.tw_fwd + (size_t)i * Sh::N, pc, ld, st, x);
    const u64 *accp = a.accq + (((size_t)c * 2 + k) * n + i) * Sh::N;
    u64 *out = a.out + (((size_t)c * 2 + k) * n + i) * Sh::N;
    sub_scale_run<Sh>(x, accp, lc.R, lc.R_sh, pc, m, tid);
    store_run<Sh>(out, x, m, tid);
}

// RS, first half: y_k = INTT_{q_l}(c_k[q_l]) -> lift2 (coefficient domain).
template <int LOG_B, int LOG_C, int LOG_E>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E>::MIN_CTAS)
k_rs_lift(EvalArgs a)
{
    stream_order();
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    extern __shared__ __align__(16) u64 smem[];
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    const u32 item = blockIdx.x >> LOG_C;
    const u32 n = a.n, l = n - 1;
    const u32 c = item / 2, k = item % 2;
    const PrimeConst pc = a.ctx.pc[l];
    const u64 *src = a.ct2 + (((size_t)c * 2 + k) * n + l) * Sh::N;
    u64 *dst = a.lift2 + ((size_t)c * 2 + k) * Sh::N;
    u64 x[Sh::E];
    auto ld = [&](u32 P) -> u64 { return rd(src + P); };
    auto st = [&](u32 P, u64 v) { dst[P] = v; };
    ntt_inv_block<Sh, false>(smem, m, 0, a.ctx.tw_inv + (size_t)l * Sh::N, pc, ld, st, x);
}

// RS, second half: out[c][k][i] = (c_k[q_i] - NTT(r mod q_i)) q_l^-1, i < l.
template <int LOG_B, int LOG_C, int LOG_E>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E>::MIN_CTAS)
k_rs(EvalArgs a)
{
    stream_order();
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    extern __shared__ __align__(16) u64 smem[];
    const u32 tid = threadIdx.x;
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    const u32 item = blockIdx.x >> LOG_C;
    const u32 n = a.n, l = n - 1;
    const u32 c = item / (2 * l), k = (item / l) % 2, i = item % l;
    const PrimeConst pc = a.ctx.pc[i];
    const DropConst dc = a.ctx.drop[(size_t)l * a.ctx.n_data + i];
    const u64 half_l = (a.ctx.pc[l].p - 1) / 2;
    const u64 *y = a.lift2 + ((size_t)c * 2 + k) * Sh::N;
    u64 x[Sh::E];
    auto ld = [&](u32 P) -> u64 { return centred_mod(rd(y + P), half_l, dc.ql, pc); };
    auto st = [&](u32, u64) {};
    ntt_fwd_block<Sh, false>(smem, m, 0, a.ctx.tw_fwd + (size_t)i * Sh::N, pc, ld, st, x);
    const u64 *src = a.ct2 + (((size_t)c * 2 + k) * n + i) * Sh::N;
    u64 *out = a.out + (((size_t)c * 2 + k) * l + i) * Sh::N;
    sub_scale_run<Sh>(x, src, dc.ql_inv, dc.ql_inv_sh, pc, m, tid);
    store_run<Sh>(out, x, m, tid);
}

// MulLinRS after the mod-up: mod-down by P and rescale by q_l. The transform
// is linear, so both divisions of limb i < l share one:
//   out_i = (d + (acc_i - NTT_i(r_P)) P^-1 - NTT_i(r_l)) q_l^-1
//         = (s_i - NTT_i((r_P P^-1 + r_l) 2^-64)) 2^64 q_l^-1    (mod q_i)
// with s the stored (acc P^-1 + d) 2^-64, r_P the centred residue of y_P =
// INTT_P(acc) and r_l that of the relinearised limb q_l, which is needed in
// the coefficient domain only:
//   y_l = INTT_l(d + (acc_l - NTT_l(r_P)) P^-1) = INTT_l(2^64 s_l) - r_P P^-1.
// So limb q_l takes one inverse transform like the special prime (both in
// k_mrr_lift; 2^64 is folded into its N^-1 constants), and the 2 (n - 1)
// forward transforms of k_mrr_rest form r_P P^-1 + r_l on their loads. Against
// a forward and an inverse transform for limb q_l and two forward transforms
// for every other limb this leaves 2 + 2 + 2 (n - 1) transforms of
// 2 + 4 + 4 (n - 1). The outputs are canonical, so they are the same words.
// Measured by itself (one context with 7 + 1 primes at N = 2^14, level 6): 64
// pairs 1157 -> 1005 us, one pair 104 -> 75 us.

// (r_P P^-1 + r_l) 2^-64 mod q_i as a transform input below 7 q_i, from y_P
// and a_l = INTT_l(2^64 s_l) (both canonical): with b_P, b_l the flags of the
// residues above half,
//   y_l = a_l - y_P P^-1 + b_P (mod q_l),
//   r_P P^-1 + r_l = y_P P^-1 + (y_l - b_P) - b_l q_l (mod q_i).
struct RestLift {
    u64 half_P, half_l, ql;
    u64 Pinv_l, Pinv_l_sh;   // P^-1 mod q_l
    u64 k1, k1_sh, k2, k2_sh;
    u64 minus_ql_k2;
    __device__ __forceinline__ u64 operator()(u64 yP, u64 al, const PrimeConst &pc) const
    {
        const u64 bP = yP > half_P ? 1u : 0u;
        const u64 yl = reduce_once(sub_mod(al, mul_shoup(yP, Pinv_l, Pinv_l_sh, ql), ql) + bP, ql);
        const u64 t0 = reduce_once(mul_shoup_lazy4_asm(yP, k1, k1_sh, pc.neg_p), pc.two_p);   // below 2 q_i
        const u64 t1 = mul_shoup_lazy4_asm(yl + pc.p - bP, k2, k2_sh, pc.neg_p);              // below 4 q_i
        return t0 + t1 + (yl > half_l ? minus_ql_k2 : 0);
    }
};

// item = 2 l c + l k + i (ciphertext c, component k, limb i < l).
template <class Sh>
__device__ __forceinline__ void mrr_rest_body(const EvalArgs &a, u32 item, u32 m, u32 rbase, bool valid)
{
    extern __shared__ __align__(16) u64 smem[];
    const u32 tid = threadIdx.x;
    const u32 n = a.n, l = n - 1, nd = a.ctx.n_data;
    const u32 c = item / (2 * l), k = (item / l) % 2, i = item % l;
    const PrimeConst pc = a.ctx.pc[i];
    const DropConst &dc = a.ctx.drop[(size_t)l * nd + i];
    const LimbConst &lc = a.ctx.limb[i];
    RestLift lift;
    lift.half_P = (a.ctx.pc[nd].p - 1) / 2;
    lift.ql = a.ctx.pc[l].p;
    lift.half_l = (lift.ql - 1) / 2;
    lift.Pinv_l = a.ctx.limb[l].Pinv;
    lift.Pinv_l_sh = a.ctx.limb[l].Pinv_sh;
    lift.k1 = lc.k1;
    lift.k1_sh = lc.k1_sh;
    lift.k2 = lc.k2;
    lift.k2_sh = lc.k2_sh;
    lift.minus_ql_k2 = dc.minus_ql_k2;
    const u64 C = dc.R_ql_inv, C_sh = dc.R_ql_inv_sh;
    const u64 *yP = a.plift + ((size_t)c * 2 + k) * Sh::N;
    const u64 *al = a.lift2 + ((size_t)c * 2 + k) * Sh::N;
    u64 x[Sh::E];
    auto nost = [&](u32, u64) {};
    auto ld = [&](int P) -> u64 { return lift(rd(yP + P), rd(al + P), pc); };
    ntt_fwd_block<Sh, false, true>(smem, m, rbase, a.ctx.tw_fwd + (size_t)i * Sh::N, pc, ld, nost, x);
    const u64 *accp = a.accq + (((size_t)c * 2 + k) * n + i) * Sh::N;
    u64 *out = a.out + (((size_t)c * 2 + k) * l + i) * Sh::N;
    sub_scale_run<Sh>(x, accp, C, C_sh, pc, m, tid);
    if (valid) store_run<Sh>(out, x, m, tid);
}

// Inverse transforms before the rest: items below 2 count take accq's limb l
// of row item = 2 c + k to lift2, times 2^64 (the lift constants); the next
// 2 count take the special-prime rows of plift in place (inputs in [0, 4P),
// the key multiply-accumulate's range; not launched after the fused mod-up,
// which leaves them transformed). Every load precedes the cluster barrier
// before the cross-CTA stages (or, in one CTA, the barrier of the first
// round exchange) and every store follows it, so a row can be transformed in
// place.
template <class Sh>
__device__ __forceinline__ void mrr_lift_body(const EvalArgs &a, u32 item, u32 m, u32 rbase, bool valid)
{
    extern __shared__ __align__(16) u64 smem[];
    const u32 n = a.n, l = n - 1;
    const bool special = item >= 2 * a.count;
    const u32 row = special ? item - 2 * a.count : item;
    const u32 pr = special ? a.ctx.n_data : l;
    const PrimeConst pc = a.ctx.pc_lift[pr];
    const u64 *src = special ? a.plift + (size_t)row * Sh::N : a.accq + ((size_t)row * n + l) * Sh::N;
    u64 *dst = (special ? a.plift : a.lift2) + (size_t)row * Sh::N;
    const u32 tid = threadIdx.x;
    u64 x[Sh::E];
#pragma unroll
    for (int e = 0; e < Sh::E; e += 4) ld4(src + last_pos<Sh>(m, tid, e), x[e], x[e + 1], x[e + 2], x[e + 3]);
    auto nold = [&](u32) -> u64 { return 0; };
    auto st = [&](u32 P, u64 v) {
        if (valid) dst[P] = v;
    };
    ntt_inv_block<Sh, true>(smem, m, rbase, a.ctx.tw_inv + (size_t)pr * Sh::N, pc, nold, st, x);
}

template <int LOG_B, int LOG_C, int LOG_E, bool JOBS = false>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E>::MIN_CTAS)
k_mrr_lift(EvalArgs a0, JobsArg<JOBS> tab)
{
    stream_order();
    EvalArgs a = a0;
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    u32 item = blockIdx.x >> LOG_C;
    if constexpr (JOBS) item = bind_job(a, tab, JS_LIFT, item);
    mrr_lift_body<Sh>(a, item, m, 0, true);
}

template <int LOG_B, int LOG_C, int LOG_E, bool JOBS = false>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E>::MIN_CTAS)
k_mrr_rest(EvalArgs a0, JobsArg<JOBS> tab)
{
    stream_order();
    EvalArgs a = a0;
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    u32 item = blockIdx.x >> LOG_C;
    if constexpr (JOBS) item = bind_job(a, tab, JS_REST, item);
    mrr_rest_body<Sh>(a, item, m, 0, true);
}

// Encryption (Sec. II-A): the transforms of the small random polynomials,
// out[c][w][l] = NTT_l(x mod q_l) for w = 0, 1, 2 (v, e0, e1 of message c; |x| <
// q_l), formed on the loads from the given draws or from the seed. Item =
// (3 c + w) n + l. Five messages of 7 limbs at N = 2^14 (105 transforms): a
// noise pass and the transforms took 11 + 24 us, 25 us this way.
template <int LOG_B, int LOG_C, int LOG_E>
__global__ void __launch_bounds__(NttShape<LOG_B, LOG_C, LOG_E>::T, NttShape<LOG_B, LOG_C, LOG_E>::MIN_CTAS)
k_enc_noise(EvalArgs a)
{
    stream_order();
    using Sh = NttShape<LOG_B, LOG_C, LOG_E>;
    extern __shared__ __align__(16) u64 smem[];
    const u32 m = (LOG_C > 0) ? cluster_ctarank() : 0u;
    const u32 item = blockIdx.x >> LOG_C;
    const u32 l = item % a.n, w = (item / a.n) % 3, c = item / (3 * a.n);
    const PrimeConst pc = a.ctx.pc[l];
    const int8_t *src = a.v ? (w == 0 ? a.v : (w == 1 ? a.e0 : a.e1)) + (size_t)c * Sh::N : nullptr;
    auto ld = [&](int P) -> u64 {
        const int x = src ? src[P] : enc_draw(a.seed, w, c, (u64)P, Sh::LOG_N);
        return x >= 0 ? (u64)x : pc.p - (u64)(-x);
    };
    auto nost = [&](u32, u64) {};
    u64 x[Sh::E];
    ntt_fwd_block<Sh>(smem, m, 0, a.ctx.tw_fwd + (size_t)l * Sh::N, pc, ld, nost, x);
    store_run<Sh>(a.out + (size_t)item * Sh::N, x, m, threadIdx.x);
}

}  // namespace he
