// launch.h -- argument blocks of the kernels and the per-degree launcher
// table (host and device visible). Internal to the library.
#pragma once
#include <cuda.h>   // CUtensorMap (the type only; nothing links the driver library)
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <type_traits>

#include "modarith.cuh"

namespace he {

// Launches of this library may begin when the CTAs of the kernel ahead of them
// in the stream have exited, before that grid is flushed and retired
// (programmatic dependent launch): the launch latency overlaps its end. Every
// kernel launched this way calls stream_order() before it touches memory, which
// waits until everything ahead in the stream is complete and visible. What a
// kernel reads that an earlier kernel may have written goes through coherent
// loads (a load through the read-only path could move ahead of the wait);
// tables and keys, written before their handle existed, may use it.
// Measured between the five launches of one MulLinRS at N = 2^14: 61 -> 43 us;
// three launches of an encryption 43 -> 36 us. Letting the next grid start
// earlier (griddepcontrol.launch_dependents) places its CTAs on the SMs the
// running grid leaves free, several on one: 9 x 3 products at 2^13 23 -> 35 us.
#ifdef __CUDACC__
__device__ __forceinline__ void stream_order()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class K, class... Args>
static cudaError_t launch_k(K kernel, u32 grid, u32 block, u32 smem, u32 cluster, cudaStream_t s, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cluster > 1) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = cluster;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
    // a refused launch is reported here and not by a later call's check as well
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}
#endif

// One limb of a batched transform (plans): its data, twiddles and constants.
struct LimbJob {
    u64 *data;
    const ulonglong2 *tw_fwd;
    const ulonglong2 *tw_inv;
    const PrimeConst *pc;
};

// A uniform batch (items = count * limbs limbs of one degree, limb l of each
// polynomial using prime first_prime + l of one table set), or a job list.
// tma_store: the forward transform writes its output with bulk tensor
// stores through tmap, the batch viewed as rows of 16 words (128 bytes),
// boxes of 32 rows, 128-byte swizzle (uniform batches, 16 words a thread).
// src: the inverse transform reads its input there instead (same layout,
// null: in place).
struct NttLaunch {
    u64 *base;
    const u64 *src;
    u32 limbs;
    u32 first_prime;
    u32 items;
    u32 prefetch;               // > 0: each cluster asks L2 for the limb this many items ahead
    const ulonglong2 *tw_fwd;   // [prime][N]
    const ulonglong2 *tw_inv;
    const PrimeConst *pc;       // [prime]
    const LimbJob *jobs;        // non-null: per-item jobs instead of base/limbs
    u32 tma_store;
    CUtensorMap tmap;
};

// Fused negacyclic product c = a b mod (X^N + 1, q) of items = count * limbs
// limbs (limb l of polynomial p at (p limbs + l) N, prime first_prime + l):
// forward transforms of a and b, pointwise product and inverse transform in
// one launch, the data staying on chip in between.
struct NegaLaunch {
    u64 *c;
    const u64 *a, *b;
    u32 limbs;
    u32 items;
    const ulonglong2 *tw_fwd;   // [prime][N]
    const ulonglong2 *tw_inv;
    const PrimeConst *pc;       // [prime]
};

// A unit of the mixed-degree transform: up to 8 >> (log_n - 12)
// limbs of degree 2^log_n, jobs[first_job .. first_job + n_jobs).
struct MixedUnit {
    u32 log_n;
    u32 first_job;
    u32 n_jobs;
    u32 pad;
};

// Mixed-degree transform of N in [2^12, 2^15]: one launch of `clusters`
// clusters of 8 CTAs walking the unit list (mixed.cu; plans launch one
// cluster per unit).
cudaError_t launch_ntt_mixed(const MixedUnit *units, u32 n_units, const LimbJob *jobs, bool inverse, u32 clusters,
                             cudaStream_t s);

// Constants of data prime q_i for the divisions. The mod-up leaves its
// accumulators on the data primes divided by P, with d_k added, and scaled by
// 2^-64 (the Montgomery reduction of its sums): k1 and k2 bring the lift of
// the special prime's rows to that scale, R takes it off again.
struct LimbConst {
    u64 Pinv, Pinv_sh;   // P^-1 mod q_i
    u64 k1, k1_sh;       // P^-1 2^-64
    u64 k2, k2_sh;       // 2^-64
    u64 R, R_sh;         // 2^64
};
// Constants of dropping q_l, for the remaining limb q_i.
struct DropConst {
    u64 ql_inv, ql_inv_sh;   // q_l^-1 mod q_i
    u64 ql;                  // q_l mod q_i
    u64 R_ql_inv, R_ql_inv_sh;   // 2^64 q_l^-1
    u64 minus_ql_k2;         // -q_l 2^-64
};

// Device view of a modulus chain (q_0..q_{n_data-1}, then P at n_data).
struct DevCtx {
    const ulonglong2 *tw_fwd;   // [n_data + 1][N]
    const ulonglong2 *tw_inv;
    const PrimeConst *pc;       // [n_data + 1]
    const PrimeConst *pc_lift;  // pc, the data primes' last inverse stage also multiplying by 2^64
    const LimbConst *limb;      // [n_data]
    const DropConst *drop;      // [l][n_data], i < l
    u32 N;
    u32 n_data;
};

// Input of a key switch: a pair of ciphertexts to multiply, a three-component
// ciphertext, or a rotation.
enum SourceKind { SRC_PAIR = 0, SRC_THREE, SRC_ROTATE, SRC_ANY };

struct EvalArgs {
    const u64 *ct_a, *ct_b;     // [count][2][n][N] (fused Mul) or null
    const u64 *ct3;             // [count][3][n][N] or null; with galois, [count][2][n][N]
    const u64 *ct2;             // [count][2][n][N] rescale input
    u64 *out;
    u64 *c2;                    // scratch [count][n][N]
    u64 *accq;                  // scratch [count][2][n][N]
    u64 *plift;                 // scratch [count][2][N]
    u64 *lift2;                 // scratch [count][2][N]
    // key words [n_data][2][n_data + 1][N]: value P^-1 mod q_i (2^64 P^-1 for digit
    // j = i), value 2^64 mod P on the special prime; and their Shoup quotients
    const u64 *evk_mac, *evk_sh;
    u64 *mx;                    // expanded mod-up scratch [group][n + 1][n][N]
    u32 n;                      // limbs at the current level
    u32 count;
    u32 c_first;                // first ciphertext of the expanded mod-up group
    // randomness of an encryption: the draws [count][N], or (v null) the seed
    // they come from
    const int8_t *v, *e0, *e1;
    u64 seed;
    u32 galois;                 // nonzero: the input is (sigma(c0), 0, sigma(c1)), sigma: X -> X^galois
    DevCtx ctx;
};

// Mixed-level batches (one context): each launch of the MulLinRS pipeline
// covers every job; job i's items in stage S start at job[i].begin[S].
// Multi-degree batches (a context and key per job, degrees 2^12 .. 2^15):
// the transform stages count units (clusters of 8 CTAs, each running 8 >> c
// items of degree 2^(12 + c) side by side) instead of items. JS_MAC counts
// tiles of MAC_BLOCK positions.
enum JobStage { JS_DIGITS = 0, JS_EXPAND, JS_MAC, JS_LIFT, JS_REST, JS_COUNT };
constexpr u32 kMaxJobs = 16;
struct EvalJob {
    const u64 *ct_a, *ct_b;     // [count][2][n][N]
    u64 *out;                   // [count][2][n - 1][N]
    u64 *c2, *accq, *plift, *lift2, *mx;   // the job's scratch regions
    const u64 *evk_mac;         // the job's key
    DevCtx ctx;                 // the job's context
    u32 n, count;
    u32 begin[JS_COUNT];
};
struct JobTable {               // passed by value (kernel parameter space)
    EvalJob job[kMaxJobs];
    u32 n_jobs;
};
struct NoJobs {};
template <bool JOBS>
using JobsArg = typename std::conditional<JOBS, JobTable, NoJobs>::type;

// Stages of the multi-degree MulLinRS pipeline (multi.cu), one launch each
// over `units` clusters; the key multiply-accumulate between the expansion
// and the lifts is k_ks_mac over the same job table.
enum MultiStage { MS_DIGITS = 0, MS_EXPAND, MS_LIFT, MS_REST, MS_COUNT };
cudaError_t launch_mrr_multi(MultiStage stage, const EvalArgs &a, const JobTable &t, u32 units, cudaStream_t s);

enum EvalKernel {
    EK_KS_DIGITS = 0,   // by the source: pair (also job tables), three components, rotation
    EK_KS_DIGITS_THREE,
    EK_KS_DIGITS_ROTATE,
    EK_KS_MODUP,
    EK_KS_EXPAND,
    EK_KS_MODDOWN,
    EK_RS_LIFT,
    EK_RS,
    EK_MRR_LIFT,
    EK_MRR_REST,
    EK_ENC_NOISE,
    EK_COUNT
};

// Launchers of one polynomial degree N = 2^log_n. A transform shape is
// (log_b, log_e): 2^log_b words per CTA (a cluster of N / 2^log_b CTAs per
// limb) and 2^log_e words per thread (radix-2^log_e register rounds); 0, 0
// picks the degree's default shape.
struct DegreeOps {
    int log_n;
    int default_log_b;
    int default_log_e;
    // Plain transform of a uniform batch or a job list, one cluster per limb.
    cudaError_t (*ntt)(const NttLaunch &a, int log_b, int log_e, bool inverse, cudaStream_t s);
    // Persistent transform over a job list with `grid_clusters` clusters.
    cudaError_t (*ntt_persistent)(const NttLaunch &a, int log_b, int log_e, bool inverse, u32 grid_clusters,
                                  cudaStream_t s);
    // Largest number of co-resident clusters of the persistent kernel.
    int (*max_clusters)(int log_b, int log_e, bool inverse);
    // Evaluation kernels over `items` clusters (the default words per CTA;
    // log_e = 3 or 4 words per thread, 0 = 4); with a job table (MulLinRS
    // kernels only) the items run over every job of a mixed-level batch.
    cudaError_t (*eval)(EvalKernel k, const EvalArgs &a, u32 items, int log_e, const JobTable *jobs,
                        cudaStream_t s);
    // Is the shape built for this degree?
    bool (*has_shape)(int log_b, int log_e);
    // Fused negacyclic product in the given transform shape (0, 0 = default).
    cudaError_t (*negacyclic)(const NegaLaunch &a, int log_b, int log_e, cudaStream_t s);
    // Its clusters that fit on the GPU together (0: the shape cannot be placed).
    int (*negacyclic_clusters)(int log_b, int log_e);
    // Shapes built for this degree: n pairs (log_b, log_e), default first.
    int n_shapes;
    const int (*shapes)[2];
};

const DegreeOps *degree_ops(int log_n);

// Encoding and decoding (encode.cu): the slot FFT of n = N/2 points in two
// passes (n = n1 n2, n1 = 2^log_n1), fused with the slot permutation and
// scaling at one end and the twist by zeta^k at the other.
struct FftArgs {
    const double2 *z_in;     // encode: slots [count][n]
    double2 *z_out;          // decode: slots [count][n]
    const double *m_in;      // decode: centred coefficients [count][N]
    u64 *pt_out;             // encode: coefficient residues [count][limbs][N]
    double2 *u;              // scratch between the passes [count][n]
    const double2 *omega;    // exp(-2 pi i j / n), j < n
    const double2 *zeta;     // exp(i pi k / N), k < n
    const u32 *slot_of;      // slot j of FFT index t_j = (5^j mod 2N - 1) / 4
    const u64 *primes;       // encode: (q_i, floor(2^64 / q_i)), i < limbs
    double scale;            // encode: Delta; decode: 1 / Delta
    double inv_n;            // 1 / n
    u32 log_n, log_n1, limbs, count;
};
cudaError_t launch_encode_fft(const FftArgs &a, cudaStream_t s);
cudaError_t launch_decode_fft(const FftArgs &a, cudaStream_t s);
// Words of the CRT kernel's multi-word integers for `need` words (0: too many).
u32 crt_words(u32 need);
cudaError_t launch_crt_compose(double *out, const u64 *coef, const u64 *tab, const u64 *primes, u32 nw, u32 log_N,
                               u32 limbs, u64 total, u32 blocks, cudaStream_t s);

}  // namespace he
