// Instantiates the bit-sliced filter kernels for one decider set PF_SLICE_D (see
// SliceWalk: 1, 5, 6 or 7).
#include <algorithm>

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

#if PF_SLICE_D != 5   // (the grids of 1 serve it)
const void *PF_CAT(sliced_ptr_, PF_SLICE_D)(int cfg) {
    return reinterpret_cast<const void *>(sliced_at<0>(cfg));
}
#endif

cudaError_t PF_CAT(launch_sliced_, PF_SLICE_D)(int cfg, int grid, const BatchArgs &b, int bin,
                                               cudaStream_t st) {
    const KernelCfg &c = kBatchCfgs[cfg];
    SliceFn f = sliced_at<0>(cfg);
    if (!f) return cudaErrorInvalidValue;
    f<<<grid, cfg_threads(c, 1), slice_smem_bytes(c.tpp, b), st>>>(b, bin, c.xe);
    return cudaGetLastError();
}

template <int L>
static cudaError_t launch_small_l(const BatchArgs &b, const SliceBins &bins, int single, int sms,
                                  cudaStream_t st) {
    const int64_t tile = 32 * (32 / L);
    const int64_t tiles = (b.f.n + tile - 1) / tile + (single < 0 ? PF_MAX_E : 0);
    const int64_t grid = std::min<int64_t>(tiles, (int64_t)sms * 32);
    filter_sliced_small_kernel<L, PF_SLICE_D>
        <<<(unsigned)grid, 32, slice_smem_bytes(L, b), st>>>(b, bins, single);
    return cudaGetLastError();
}

cudaError_t PF_CAT(launch_small_, PF_SLICE_D)(int lanes, const BatchArgs &b, const SliceBins &bins,
                                              int single, int sms, cudaStream_t st) {
    switch (lanes) {
        case 8: return launch_small_l<8>(b, bins, single, sms, st);
        case 16: return launch_small_l<16>(b, bins, single, sms, st);
    }
    return cudaErrorInvalidValue;
}

template <int CLS>
static cudaError_t launch_bins_c(int cls, const BatchArgs &b, const SliceBins &bins, int sms,
                                 cudaStream_t st) {
    if (cls == CLS) {
        constexpr int DPT = (kSliceClassE[CLS] + 2) / 2;
        filter_sliced_bins_kernel<DPT, PF_SLICE_D>
            <<<slice_warps(DPT, PF_SLICE_D & 2) * sms, 32, slice_smem_bytes(4, b), st>>>(b, bins);
        return cudaGetLastError();
    }
    if constexpr (CLS + 1 < kSliceClasses) return launch_bins_c<CLS + 1>(cls, b, bins, sms, st);
    return cudaErrorInvalidValue;
}

cudaError_t PF_CAT(launch_slice_bins_, PF_SLICE_D)(int cls, const BatchArgs &b,
                                                   const SliceBins &bins, int sms,
                                                   cudaStream_t st) {
    return launch_bins_c<0>(cls, b, bins, sms, st);
}

}  // namespace pf
