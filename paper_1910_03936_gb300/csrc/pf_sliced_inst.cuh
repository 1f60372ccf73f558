// Instantiates the bit-sliced filter kernels for one decider set PF_SLICE_D (see
// SliceWalk: 1, 5, 6 or 7).
#include "pf_sliced.cuh"

namespace pf {

#define PF_CAT2(a, b) a##b
#define PF_CAT(a, b) PF_CAT2(a, b)

using SliceFn = void (*)(BatchArgs, int, int);

template <int I>
static SliceFn sliced_at(int cfg) {
    constexpr KernelCfg c = kBatchCfgs[I];
    if constexpr (cfg_sliced(c))
        if (cfg == I) return &filter_sliced_kernel<c.tpp, c.dpt, PF_SLICE_D>;
    if constexpr (I + 1 < kNumBatchCfgs) return sliced_at<I + 1>(cfg);
    return nullptr;
}

const void *PF_CAT(sliced_ptr_, PF_SLICE_D)(int cfg) {
    return reinterpret_cast<const void *>(sliced_at<0>(cfg));
}

cudaError_t PF_CAT(launch_sliced_, PF_SLICE_D)(int cfg, int grid, const BatchArgs &b, int bin,
                                               cudaStream_t st) {
    const KernelCfg &c = kBatchCfgs[cfg];
    SliceFn f = sliced_at<0>(cfg);
    if (!f) return cudaErrorInvalidValue;
    f<<<grid, cfg_threads(c, 1), cfg_smem(c, 1), st>>>(b, bin, c.xe);
    return cudaGetLastError();
}

}  // namespace pf
