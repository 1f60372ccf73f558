// Host-side table of the filter kernel configurations and the launchers of
// every kernel in the library.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "pf_internal.cuh"

namespace pf {

// One batched-filter configuration: TPP lanes per pair, DPT diagonal slots
// per lane; it serves thresholds E <= ecap.  xe >= 0 marks the
// exact-threshold form (one thread per pair, serves E == xe only).  words
// > 0 marks its two-phase form: the mask words of pairs up to `words`
// 32-column words are kept in shared memory and SneakySnake runs as a
// per-lane step loop over them (longer pairs take the fused loop).
// sliced marks a bit-sliced configuration (pf_sliced.cuh): tpp lanes share 32
// pairs of threshold xe with dpt diagonals each.
struct KernelCfg {
    int tpp, dpt, ecap, xe, words;
    bool sliced = false;
};

constexpr KernelCfg kBatchCfgs[] = {
    {1, 4, 3, -1},   {2, 4, 3, -1},   {4, 2, 3, -1},   {8, 1, 3, -1},
    {1, 8, 7, -1},   {2, 8, 7, -1},   {4, 4, 7, -1},   {8, 2, 7, -1},  {16, 1, 7, -1},
    {1, 16, 15, -1}, {2, 16, 15, -1}, {4, 8, 15, -1},  {8, 4, 15, -1}, {16, 2, 15, -1},
    {32, 1, 15, -1},
    {2, 32, 31, -1}, {4, 16, 31, -1}, {8, 8, 31, -1},  {16, 4, 31, -1}, {32, 2, 31, -1},
    {1, 1, 0, 0},    {1, 2, 1, 1},    {1, 3, 2, 2},    {1, 4, 3, 3},   {1, 5, 4, 4},
    {1, 6, 5, 5},    {1, 7, 6, 6},    {1, 8, 7, 7},    {1, 9, 8, 8},   {1, 10, 9, 9},
    {1, 11, 10, 10}, {1, 12, 11, 11}, {1, 13, 12, 12}, {1, 14, 13, 13}, {1, 15, 14, 14},
    {1, 16, 15, 15},
    // two-phase forms, E = 1..12: as many words as keep a 4-warp block's
    // arrays within about 56 KB (four blocks per SM)
    {1, 2, 1, 1, 8},     {1, 3, 2, 2, 8},     {1, 4, 3, 3, 8},     {1, 5, 4, 4, 8},
    {1, 6, 5, 5, 8},     {1, 7, 6, 6, 8},     {1, 8, 7, 7, 7},     {1, 9, 8, 8, 6},
    {1, 10, 9, 9, 5},    {1, 11, 10, 10, 5},  {1, 12, 11, 11, 4},  {1, 13, 12, 12, 4},
    // and with 5-word arrays (pairs up to 160 bases) for E = 1..7: smaller
    // blocks, more of them per SM,
    {1, 2, 1, 1, 5},     {1, 3, 2, 2, 5},     {1, 4, 3, 3, 5},     {1, 5, 4, 4, 5},
    {1, 6, 5, 5, 5},     {1, 7, 6, 6, 5},     {1, 8, 7, 7, 5},
    // and for E = 11..15 (up to 79 KB per block, two or three per SM)
    {1, 12, 11, 11, 5},  {1, 13, 12, 12, 5},  {1, 14, 13, 13, 5},  {1, 15, 14, 14, 5},
    {1, 16, 15, 15, 5},
    // two-phase forms with a lane group per pair (pairs up to 256 bases): for
    // thresholds whose masks do not fit one thread
    {4, 4, 7, -1, 8},    {4, 8, 15, -1, 8},   {8, 4, 15, -1, 8},   {4, 16, 31, -1, 8},
    {8, 8, 31, -1, 8},   {16, 4, 31, -1, 8},
    // fewer slots per lane, fewer dead ones: 56 slots for E <= 27, 48 for
    // E <= 23, 40 for E <= 19
    {8, 7, 27, -1, 8},   {8, 6, 23, -1, 8},   {8, 5, 19, -1, 8},
    // one thread per pair with 8-word arrays (pairs up to 256 bases) for
    // E = 8..13: 68 KB (three blocks per SM) to 108 KB (two) per block
    {1, 9, 8, 8, 8},     {1, 10, 9, 9, 8},    {1, 11, 10, 10, 8},  {1, 12, 11, 11, 8},
    {1, 13, 12, 12, 8},  {1, 14, 13, 13, 8},
    // lane groups of two and four (fewer shuffles per step, the walk's
    // control repeated by fewer lanes): the fastest at E = 16..31
    {2, 17, 16, -1, 8},  {4, 11, 21, -1, 8},  {4, 13, 25, -1, 8},  {2, 26, 25, -1, 8},
    // bit-sliced, one threshold each: E = 5..27 with four lanes per group (at
    // E = 20 and 25 eight lanes were no faster: 0.54 against 0.52 and 0.63
    // against 0.57 ms per 2M pairs of 250 bp with both deciders), E = 28..31
    // with eight (more diagonals per lane than registers hold)
    {4, 3, 5, 5, 0, true}, {4, 4, 6, 6, 0, true}, {4, 4, 7, 7, 0, true},
    {4, 5, 8, 8, 0, true}, {4, 5, 9, 9, 0, true}, {4, 6, 10, 10, 0, true},
    {4, 6, 11, 11, 0, true}, {4, 7, 12, 12, 0, true}, {4, 7, 13, 13, 0, true},
    {4, 8, 14, 14, 0, true}, {4, 8, 15, 15, 0, true}, {4, 9, 16, 16, 0, true},
    {4, 9, 17, 17, 0, true}, {4, 10, 18, 18, 0, true}, {4, 10, 19, 19, 0, true},
    {4, 11, 20, 20, 0, true}, {4, 11, 21, 21, 0, true}, {4, 12, 22, 22, 0, true},
    {4, 12, 23, 23, 0, true}, {4, 13, 24, 24, 0, true}, {4, 13, 25, 25, 0, true},
    {4, 14, 26, 26, 0, true}, {4, 14, 27, 27, 0, true}, {8, 8, 28, 28, 0, true},
    {8, 8, 29, 29, 0, true}, {8, 8, 30, 30, 0, true}, {8, 8, 31, 31, 0, true},
};

constexpr bool cfg_sliced(const KernelCfg &c) { return c.sliced; }

// A bit-sliced warp's tile: columns per block of the walk, words per segment
// and words of shared memory (SliceColumns).
__host__ __device__ constexpr int slice_block(int L) { return L >= 8 ? 8 : 4; }
__host__ __device__ constexpr int slice_seg(int L) { return L / 4; }
__host__ __device__ constexpr size_t slice_smem_words(int L) {
    return (size_t)3 * (32 / L) *
           (32 * (slice_seg(L) + 2) + slice_block(L) - 1 + 32 * slice_seg(L));
}
// A side whose words are found by an unsigned 32-bit step from pair to pair (rows
// may also run backwards: pf_filter_partitioned takes negative strides).
__host__ __device__ constexpr bool slice_strided(const SeqView &v) {
    return !v.off && v.stride >= 0 && v.stride < (1 << 24);
}
// and the bytes with the starts of its pairs where the launch needs them (the
// smaller, the more L1 is left for the loads: 0.36 against 0.39 ms for 4M pairs
// of 150 bp at E = 6 without the two tables)
inline size_t slice_smem_bytes(int L, const BatchArgs &b) {
    const SeqView &r = b.f.pairs.read, &f = b.f.pairs.ref;
    const bool strided = !b.order && slice_strided(r) && slice_strided(f);
    const int tables = strided ? 0 : (r.off == f.off && r.stride == f.stride ? 1 : 2);
    return slice_smem_words(L) * sizeof(uint32_t) + tables * 32 * (32 / L) * sizeof(int64_t);
}
// Words of the longest pair that the layout allows: strided rows hold no more
// (rows that overlap or repeat tell nothing).
inline int64_t row_words(const PairsView &pv) {
    const SeqView &r = pv.read, &f = pv.ref;
    const int64_t lo = r.stride < f.stride ? r.stride : f.stride;
    return r.off || f.off || lo < 1 ? INT64_MAX : (r.stride > f.stride ? r.stride : f.stride);
}
// Warps per SM that a kernel's registers are held to.  More warps hide more
// latency but leave less L1 for the loads (the walk's arrays take 12.6 KB per
// warp, 14.6 or 16.6 with the tables of starts).  SneakySnake, 12 / 9 warps: 0.285 / 0.283 ms for 4M pairs of 150 bp at
// E = 6, 0.332 / 0.327 at E = 15, 0.382 / 0.366 for 2M of 250 bp at E = 25; with
// GateKeeper, which keeps four columns of every diagonal: E = 6 12 / 9 warps
// 0.353 / 0.359, E = 15 9 / 8 warps 0.503 / 0.535, E = 25 9 (spills) / 8 warps
// 0.666 / 0.564.
constexpr int slice_warps(int DPT, bool gatekeeper) {
    return !gatekeeper ? 9 : (DPT <= 6 ? 12 : (DPT <= 9 ? 9 : 8));
}

// Bins of several thresholds that one launch takes (launch_filter_slice_bins).
struct SliceBins {
    int count;
    unsigned char bin[32], E[32];  // rising E
};
constexpr int kSliceClassE[] = {7, 11, 15, 21, 25};  // largest threshold of each class
constexpr int kSliceClasses = 5;

// The two-phase form applies where SneakySnake runs (deciders 1 and 3);
// GateKeeper alone runs a two-phase configuration as the fused loop.
constexpr bool cfg_split(const KernelCfg &c, int dec) { return c.words > 0 && dec != 2; }
// Diagonal slots one lane stores per word in the two-phase form.
constexpr int cfg_slots(const KernelCfg &c) { return c.xe >= 0 ? 2 * c.xe + 1 : c.dpt; }
// Block size and dynamic shared memory of a configuration's kernel.
constexpr int cfg_threads(const KernelCfg &c, int dec) {
    return cfg_sliced(c) ? 32 : (cfg_split(c, dec) ? kSplitWarps * 32 : 256);
}
constexpr size_t cfg_smem(const KernelCfg &c, int dec) {
    if (cfg_sliced(c)) return slice_smem_words(c.tpp) * sizeof(uint32_t);
    return cfg_split(c, dec)
               ? (size_t)kSplitWarps * c.words * cfg_slots(c) * 32 * sizeof(uint32_t)
               : 0;
}

// Pairs one warp of a configuration's kernel takes at once: one per lane in
// the two-phase form, one per lane group in the fused loop.
constexpr int cfg_step(const KernelCfg &c, int dec) {
    return cfg_sliced(c) ? 32 * (32 / c.tpp) : 32 / c.tpp;
}

// a configuration serves threshold E
constexpr bool cfg_serves(const KernelCfg &c, int E) {
    return c.xe >= 0 ? c.xe == E : c.ecap >= E;
}
constexpr int kNumBatchCfgs = sizeof(kBatchCfgs) / sizeof(kBatchCfgs[0]);
// Inside a configuration's bin the scheduler groups pairs by length class
// (ceil(len/32) words, the last class holding 8 words and more): keys of
// the binning counting sort.
constexpr int kLenClasses = 9;
constexpr int kNumBinKeys = kNumBatchCfgs * kLenClasses;
// Work counters in the scheduler's scratch: one per configuration's bin,
// then the verifier's.
constexpr int kWorkCounters = kNumBatchCfgs + 1;
constexpr int kFirstExactCfg = 20;  // kBatchCfgs[20 + E] serves exactly E
constexpr int kTwoLaneCfg = 10, kFourLaneCfg = 16;  // E <= 15, every threshold
static_assert(kBatchCfgs[kTwoLaneCfg].tpp == 2 && kBatchCfgs[kTwoLaneCfg].ecap == 15);
static_assert(kBatchCfgs[kFourLaneCfg].tpp == 4 && kBatchCfgs[kFourLaneCfg].ecap == PF_MAX_E);
constexpr int kWideCfg = 19;        // one warp per pair, every threshold
static_assert(kBatchCfgs[kWideCfg].tpp == 32 && kBatchCfgs[kWideCfg].ecap == PF_MAX_E);

// Plain kernel (one thread per pair): DPT = kPlainDpt[i] serves E <= DPT - 1.
constexpr int kPlainDpt[] = {1, 2, 4, 8, 16, 32};
constexpr int kNumPlain = sizeof(kPlainDpt) / sizeof(kPlainDpt[0]);

// The plain kernel with the threshold fixed at compile time: E = 0..15.
constexpr int kPlainExactMaxE = 15;

// dec in {1, 2, 3}
cudaError_t launch_filter_plain(int dec, int plain_idx, const FilterArgs &a, cudaStream_t st);
cudaError_t launch_filter_plain_exact(int dec, int E, const FilterArgs &a, cudaStream_t st);
cudaError_t launch_filter_batched(int dec, int cfg, int grid, const BatchArgs &b, int bin,
                                  cudaStream_t st);
const void *filter_batched_fn(int dec, int cfg);
cudaError_t launch_filter_sliced(int dec, int cfg, int grid, const BatchArgs &b, int bin,
                                 cudaStream_t st);
const void *filter_sliced_fn(int dec, int cfg);
// One persistent launch over several bit-sliced bins (four lanes per group)
// whose thresholds belong to class cls.
cudaError_t launch_filter_slice_bins(int dec, int cls, const BatchArgs &b, const SliceBins &bins,
                                     int sms, cudaStream_t st);
// The bit-sliced kernel with more lanes per group: every pair at threshold
// `single` with 16 or (single >= 8) 8 lanes, or (single < 0) the bins with 16.
cudaError_t launch_filter_slices(int dec, int lanes, const BatchArgs &b, const SliceBins &bins,
                                 int single, int sms, cudaStream_t st);

// SneakySnake on sub-matrices (t columns, y replications), one threshold, 16 or
// four lanes per group; late: which long pairs are left out (with few, their
// counts are kLeftOut then).
constexpr int16_t kLeftOut = -2;
cudaError_t launch_submat_sliced(const FilterArgs &a, int t, int y, int lanes,
                                 const LongPairs &late, int sms, cudaStream_t st);

cudaError_t launch_pack_ragged(const uint8_t *ascii, const int64_t *byte_off,
                               const int64_t *word_off, int64_t nseq, uint32_t *lo,
                               uint32_t *hi, uint32_t *nm, unsigned *err, cudaStream_t st,
                               const int32_t *seg_of = nullptr, unsigned *seg_err = nullptr);
cudaError_t launch_pack_starts(const uint8_t *ascii, const int64_t *byte_off,
                               const int64_t *word_start, int64_t nseq, uint32_t *lo,
                               uint32_t *hi, uint32_t *nm, unsigned *err, cudaStream_t st);
cudaError_t launch_pack_fixed(const uint8_t *ascii, int64_t nseq, int len, uint32_t *lo,
                              uint32_t *hi, uint32_t *nm, unsigned *err, int sms,
                              cudaStream_t st);
int64_t compact_tiles(int64_t n);
// order (may be null; used unless *ident): position q stands for pair
// order[q], and the indices come out in that order.
cudaError_t launch_compact(const uint8_t *flags, int64_t n, int64_t *idx, int64_t *n_out,
                           int64_t *tile_scratch, cudaStream_t st,
                           const int64_t *order = nullptr, const int *ident = nullptr);
cudaError_t launch_verify(const PairsView &pv, const int32_t *lens, const int16_t *E, int E_max,
                          const int64_t *idx, const int64_t *n_idx, int64_t n, int32_t *dist,
                          unsigned *err, int sms, cudaStream_t st,
                          unsigned long long *work = nullptr, bool grouped = false);

}  // namespace pf
