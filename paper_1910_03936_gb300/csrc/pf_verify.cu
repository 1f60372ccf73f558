// a6: verification kernel, one or two pairs per thread (device functions and their
// derivation in pf_verify.cuh).
#include <algorithm>

#include "pf_verify.cuh"

namespace pf {

namespace {

// What a launch's thresholds allow: all two to a word, 32-bit bands (64-bit
// ones, SPLIT: two to a word where a chunk's thresholds do), 64-bit bands.
enum class Bands { kTwo, kOne, kSplit, kWide };

struct Slot {
    int64_t p;
    int m, E;
    bool ok;
};

__device__ __forceinline__ Slot slot_at(const int32_t *lens, const int16_t *Es, int E_max,
                                        const int64_t *idx, int64_t t, int64_t count,
                                        int32_t *dist, unsigned *err) {
    Slot s{0, 0, 0, t < count};
    if (!s.ok) return s;
    s.p = idx ? __ldg(idx + t) : t;
    s.m = __ldg(lens + s.p);
    s.E = Es ? (int)__ldg(Es + s.p) : E_max;
    if (s.m < 0 || s.E < 0 || s.E > E_max) {
        dist[s.p] = -1;
        atomicOr(err, ERR_PAIR_ARGS);
        s.ok = false;
        s.m = s.E = 0;
    }
    return s;
}

// kSplit (64-bit launches whose indices come grouped by threshold): a pair
// with E <= 15 takes the 32-bit band.  Grouped, a warp's pairs take one of
// the two; in pair order a warp would run both.
template <Bands B>
__device__ __forceinline__ void verify_one(const PairsView &pv, const Slot &s, int32_t *dist) {
    if (!s.ok) return;
    if (B == Bands::kOne || (B == Bands::kSplit && s.E <= 15))
        dist[s.p] = verify_pair<uint32_t>(pv, s.p, s.m, s.E);
    else
        dist[s.p] = verify_pair<uint64_t>(pv, s.p, s.m, s.E);
}

// A warp's chunk of positions from t0 on: one a lane, or two.
template <Bands B>
__device__ __forceinline__ void verify_chunk(const PairsView &pv, const int32_t *lens,
                                             const int16_t *Es, int E_max, const int64_t *idx,
                                             int64_t t0, int64_t count, bool two, int32_t *dist,
                                             unsigned *err) {
    const int lane = threadIdx.x & 31;
    Slot a = slot_at(lens, Es, E_max, idx, t0 + lane, count, dist, err);
    Slot b{0, 0, 0, false};
    if (two) {
        b = slot_at(lens, Es, E_max, idx, t0 + 32 + lane, count, dist, err);
        if (B == Bands::kTwo || __all_sync(0xffffffffu, max(a.E, b.E) <= kTwoE)) {
            if (!(a.ok || b.ok)) return;
            int da, db;
            verify_two(pv, a.p, b.p, a.m, b.m, a.E, b.E, da, db);
            if (a.ok) dist[a.p] = da;
            if (b.ok) dist[b.p] = db;
            return;
        }
    }
    if constexpr (B != Bands::kTwo) {
#pragma unroll 1
        for (int k = 0; k < (two ? 2 : 1); ++k) {
            verify_one<B>(pv, a, dist);
            a = b;
        }
    }
}

// Without a work counter the warps stride over the positions.  With one
// (zeroed before the launch) they claim their chunks behind the first, which
// each has by its number, from the last position on: when the indices come
// grouped by threshold and length, the costly groups lie together at the end,
// and a fixed assignment would leave them to a few blocks.  The claims of one
// address take 2.9 ns each, so the grid is about what is resident and the next claim
// is under way while a chunk is verified: with a claim for every chunk by 1216
// blocks, 0.63M pairs of 150 bp, E = 6, took 80 us more.
template <Bands B>
__global__ void __launch_bounds__(256)
verify_kernel(PairsView pv, const int32_t *lens, const int16_t *Es, int E_max,
              const int64_t *idx, const int64_t *n_idx, int64_t n, int32_t *dist,
              unsigned *err, unsigned long long *work) {
    const int64_t count = idx ? min(*n_idx, n) : n;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const bool two = B == Bands::kTwo ||
                     ((B == Bands::kOne || B == Bands::kSplit) && Es && count >= 64 * warps);
    const int64_t chunk = two ? 64 : 32;
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t chunks = (count + chunk - 1) / chunk;
    for (int64_t item = warp; item < chunks;) {
        unsigned long long next = 0;
        if (work && (threadIdx.x & 31) == 0) next = atomicAdd(work, 1ull);
        verify_chunk<B>(pv, lens, Es, E_max, idx, (work ? chunks - 1 - item : item) * chunk, count,
                        two, dist, err);
        item = warps + (work ? (int64_t)__shfl_sync(0xffffffffu, next, 0) : item);
    }
}

// Calls from here on take two pairs to a word where all thresholds allow it.
// 2M pairs of 150 bp, E = 6: 331 us one pair a thread, 234 two; 100,000: 23.9
// and 21.7, 30,000: 11.9 and 14.0 (half as many warps, each with the longer
// columns of two pairs).
constexpr int64_t kTwoFrom = 100000;

}  // namespace

cudaError_t launch_verify(const PairsView &pv, const int32_t *lens, const int16_t *E, int E_max,
                          const int64_t *idx, const int64_t *n_idx, int64_t n, int32_t *dist,
                          unsigned *err, int sms, cudaStream_t st, unsigned long long *work,
                          bool grouped) {
    if (n <= 0) return cudaSuccess;
    const bool two = E_max <= kTwoE && n >= kTwoFrom;
    if (!E) work = nullptr;  // one threshold: no group is costlier
    // 16 to 24 warps an SM are resident (16, 20 and 24 take the same for claims);
    // striding ones come in several waves, which levels their ends (2M pairs,
    // E = 6: 64 warps an SM 5 % faster than 24).  Few pairs spread over the SMs
    // in blocks of two warps.
    const int threads = n < kTwoFrom ? 64 : 256;
    const int64_t cap = (int64_t)sms * (work ? 24 : 64) * 32 / threads;
    const int64_t per = two ? 2 * threads : threads;
    const int64_t blocks = std::min((n + per - 1) / per, cap);
    if (work) {
        const cudaError_t e = cudaMemsetAsync(work, 0, sizeof(unsigned long long), st);
        if (e != cudaSuccess) return e;
    }
    const auto kernel = two             ? verify_kernel<Bands::kTwo>
                        : E_max <= 15   ? verify_kernel<Bands::kOne>
                        : grouped && E  ? verify_kernel<Bands::kSplit>
                                        : verify_kernel<Bands::kWide>;
    kernel<<<(unsigned)blocks, threads, 0, st>>>(pv, lens, E, E_max, idx, n_idx, n, dist, err, work);
    return cudaGetLastError();
}

}  // namespace pf
