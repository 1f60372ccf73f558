// Routes a decider set to its instantiation unit.
#include "pf_kernels.h"

namespace pf {

cudaError_t launch_batched_dec1(int, int, const BatchArgs &, int, cudaStream_t);
cudaError_t launch_batched_dec2(int, int, const BatchArgs &, int, cudaStream_t);
cudaError_t launch_batched_dec3(int, int, const BatchArgs &, int, cudaStream_t);
const void *batched_fn_dec1(int);
const void *batched_fn_dec2(int);
const void *batched_fn_dec3(int);
cudaError_t launch_plain_dec1(int, const FilterArgs &, cudaStream_t);
cudaError_t launch_plain_dec2(int, const FilterArgs &, cudaStream_t);
cudaError_t launch_plain_dec3(int, const FilterArgs &, cudaStream_t);
cudaError_t launch_plain_exact_dec1(int, const FilterArgs &, cudaStream_t);
cudaError_t launch_plain_exact_dec2(int, const FilterArgs &, cudaStream_t);
cudaError_t launch_plain_exact_dec3(int, const FilterArgs &, cudaStream_t);

cudaError_t launch_sliced_1(int, int, const BatchArgs &, int, cudaStream_t);
cudaError_t launch_sliced_5(int, int, const BatchArgs &, int, cudaStream_t);
cudaError_t launch_sliced_6(int, int, const BatchArgs &, int, cudaStream_t);
cudaError_t launch_sliced_7(int, int, const BatchArgs &, int, cudaStream_t);
cudaError_t launch_small_1(int, const BatchArgs &, const SliceBins &, int, int, cudaStream_t);
cudaError_t launch_small_5(int, const BatchArgs &, const SliceBins &, int, int, cudaStream_t);
cudaError_t launch_small_6(int, const BatchArgs &, const SliceBins &, int, int, cudaStream_t);
cudaError_t launch_small_7(int, const BatchArgs &, const SliceBins &, int, int, cudaStream_t);
cudaError_t launch_slice_bins_1(int, const BatchArgs &, const SliceBins &, int, cudaStream_t);
cudaError_t launch_slice_bins_5(int, const BatchArgs &, const SliceBins &, int, cudaStream_t);
cudaError_t launch_slice_bins_6(int, const BatchArgs &, const SliceBins &, int, cudaStream_t);
cudaError_t launch_slice_bins_7(int, const BatchArgs &, const SliceBins &, int, cudaStream_t);
const void *sliced_ptr_1(int);
const void *sliced_ptr_6(int);
const void *sliced_ptr_7(int);

// SneakySnake alone counts the Hamming distance only for a caller that
// resolves distances by it.
cudaError_t launch_filter_sliced(int dec, int cfg, int grid, const BatchArgs &b, int bin,
                                 cudaStream_t st) {
    switch (dec) {
        case 1:
            return b.f.need ? launch_sliced_5(cfg, grid, b, bin, st)
                            : launch_sliced_1(cfg, grid, b, bin, st);
        case 2: return launch_sliced_6(cfg, grid, b, bin, st);
        case 3: return launch_sliced_7(cfg, grid, b, bin, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_filter_slice_bins(int dec, int cls, const BatchArgs &b, const SliceBins &bins,
                                     int sms, cudaStream_t st) {
    switch (dec) {
        case 1:
            return b.f.need ? launch_slice_bins_5(cls, b, bins, sms, st)
                            : launch_slice_bins_1(cls, b, bins, sms, st);
        case 2: return launch_slice_bins_6(cls, b, bins, sms, st);
        case 3: return launch_slice_bins_7(cls, b, bins, sms, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_filter_slices(int dec, int lanes, const BatchArgs &b, const SliceBins &bins,
                                 int single, int sms, cudaStream_t st) {
    switch (dec) {
        case 1:
            return b.f.need ? launch_small_5(lanes, b, bins, single, sms, st)
                            : launch_small_1(lanes, b, bins, single, sms, st);
        case 2: return launch_small_6(lanes, b, bins, single, sms, st);
        case 3: return launch_small_7(lanes, b, bins, single, sms, st);
    }
    return cudaErrorInvalidValue;
}

const void *filter_sliced_fn(int dec, int cfg) {
    switch (dec) {
        case 1: return sliced_ptr_1(cfg);
        case 2: return sliced_ptr_6(cfg);
        case 3: return sliced_ptr_7(cfg);
    }
    return nullptr;
}

cudaError_t launch_filter_plain_exact(int dec, int E, const FilterArgs &a, cudaStream_t st) {
    switch (dec) {
        case 1: return launch_plain_exact_dec1(E, a, st);
        case 2: return launch_plain_exact_dec2(E, a, st);
        case 3: return launch_plain_exact_dec3(E, a, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_filter_plain(int dec, int plain_idx, const FilterArgs &a, cudaStream_t st) {
    switch (dec) {
        case 1: return launch_plain_dec1(plain_idx, a, st);
        case 2: return launch_plain_dec2(plain_idx, a, st);
        case 3: return launch_plain_dec3(plain_idx, a, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_filter_batched(int dec, int cfg, int grid, const BatchArgs &b, int bin,
                                  cudaStream_t st) {
    if (cfg_sliced(kBatchCfgs[cfg])) return launch_filter_sliced(dec, cfg, grid, b, bin, st);
    switch (dec) {
        case 1: return launch_batched_dec1(cfg, grid, b, bin, st);
        case 2: return launch_batched_dec2(cfg, grid, b, bin, st);
        case 3: return launch_batched_dec3(cfg, grid, b, bin, st);
    }
    return cudaErrorInvalidValue;
}

const void *filter_batched_fn(int dec, int cfg) {
    if (cfg_sliced(kBatchCfgs[cfg])) return filter_sliced_fn(dec, cfg);
    switch (dec) {
        case 1: return batched_fn_dec1(cfg);
        case 2: return batched_fn_dec2(cfg);
        case 3: return batched_fn_dec3(cfg);
    }
    return nullptr;
}

}  // namespace pf
