// mixed.cu -- launcher of the mixed-degree transform (one launch
// for every limb of degree 2^12 .. 2^15 in a plan; see k_ntt_mixed).
#include <mutex>

#include "kernels.cuh"

namespace he {

static const u32 kMixedSmem = 4096 * 8;   // one 2^12-word block per CTA

template <bool INV>
static cudaError_t mixed_prepare()
{
    static std::once_flag f;
    static cudaError_t e = cudaSuccess;
    std::call_once(f, [] {
        e = cudaFuncSetAttribute(k_ntt_mixed<INV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMixedSmem);
    });
    return e;
}

cudaError_t launch_ntt_mixed(const MixedUnit *units, u32 n_units, const LimbJob *jobs, bool inverse, u32 clusters,
                             cudaStream_t s)
{
    if (inverse) {
        if (cudaError_t e = mixed_prepare<true>()) return e;
        return launch_k(k_ntt_mixed<true>, clusters * 8, 256, kMixedSmem, 8, s, units, n_units, jobs);
    }
    if (cudaError_t e = mixed_prepare<false>()) return e;
    return launch_k(k_ntt_mixed<false>, clusters * 8, 256, kMixedSmem, 8, s, units, n_units, jobs);
}

}  // namespace he
