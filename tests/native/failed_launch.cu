// pf_filter over fake launchers: the first launch of several is under way on a
// side stream when the next one fails.  Once the call has returned and the
// context's stream is idle, the first launch must be done as well.
#include <cstdio>
#include <vector>

#include "pf_ctx.h"
#include "pf_kernels.h"

__global__ void slow_kernel(volatile int *done) {
    unsigned x = 1u;
    for (int i = 0; i < 8000000; ++i) x = x * 1664525u + 1013904223u;   // tens of ms
    *done = x ? 1 : 2;
}

static int *g_done;
static int g_fails;

namespace pf {
cudaError_t launch_filter_slices(int, int, const BatchArgs &, const SliceBins &, int, int,
                                 cudaStream_t st) {
    slow_kernel<<<1, 1, 0, st>>>(g_done);
    return cudaGetLastError();
}
cudaError_t launch_filter_batched(int, int, int, const BatchArgs &, int, cudaStream_t) {
    ++g_fails;
    return cudaErrorInvalidValue;
}
const void *filter_batched_fn(int, int) { return reinterpret_cast<const void *>(&slow_kernel); }
// not reached
int64_t compact_tiles(int64_t n) { return (n + 4095) / 4096; }
cudaError_t launch_filter_slice_bins(int, int, const BatchArgs &, const SliceBins &, int,
                                     cudaStream_t) { return cudaErrorUnknown; }
cudaError_t launch_filter_plain(int, int, const FilterArgs &, cudaStream_t) { return cudaErrorUnknown; }
cudaError_t launch_filter_plain_exact(int, int, const FilterArgs &, cudaStream_t) { return cudaErrorUnknown; }
cudaError_t launch_compact(const uint8_t *, int64_t, int64_t *, int64_t *, int64_t *, cudaStream_t,
                           const int64_t *, const int *) { return cudaErrorUnknown; }
cudaError_t launch_verify(const PairsView &, const int32_t *, const int16_t *, int, const int64_t *,
                          const int64_t *, int64_t, int32_t *, unsigned *, int, cudaStream_t,
                          unsigned long long *, bool) { return cudaErrorUnknown; }
cudaError_t launch_pack_fixed(const uint8_t *, int64_t, int, uint32_t *, uint32_t *, uint32_t *,
                              unsigned *, int, cudaStream_t) { return cudaErrorUnknown; }
cudaError_t launch_pack_ragged(const uint8_t *, const int64_t *, const int64_t *, int64_t, uint32_t *,
                               uint32_t *, uint32_t *, unsigned *, cudaStream_t, const int32_t *,
                               unsigned *) { return cudaErrorUnknown; }
cudaError_t launch_pack_starts(const uint8_t *, const int64_t *, const int64_t *, int64_t, uint32_t *,
                               uint32_t *, uint32_t *, unsigned *, cudaStream_t) { return cudaErrorUnknown; }
}  // namespace pf
void pf_serve_teardown(pf_ctx *) {}
void pf_host_teardown(pf_ctx *) {}

int main() {
    const int n = 3000;
    pf_config cfg{0, nullptr, 0, 0u};
    pf_ctx *ctx = nullptr;
    if (pf_create(&ctx, &cfg) != PF_OK || pf_set_small_batch(ctx, 0) != PF_OK) return 2;
    char *mem = nullptr;
    if (cudaMalloc(&mem, 1 << 20) != cudaSuccess || cudaMemset(mem, 0, 1 << 20) != cudaSuccess ||
        cudaHostAlloc(&g_done, sizeof(int), cudaHostAllocMapped) != cudaSuccess)
        return 2;
    *g_done = 0;
    const pf_seqs side{reinterpret_cast<uint32_t *>(mem), reinterpret_cast<uint32_t *>(mem),
                       reinterpret_cast<uint32_t *>(mem), nullptr, 5};
    const pf_pairs pairs{side, side};
    const int32_t *lens = reinterpret_cast<int32_t *>(mem);
    const int16_t *E = reinterpret_cast<int16_t *>(mem);
    const pf_status st = pf_filter(ctx, 3u, &pairs, lens, E, 12, reinterpret_cast<uint8_t *>(mem + 65536),
                                   reinterpret_cast<int16_t *>(mem + 131072), n);
    const int at_return = *(volatile int *)g_done;
    cudaStreamSynchronize(cudaStreamPerThread);
    const int done = *(volatile int *)g_done;
    std::printf("status %d fails %d at return %d done %d\n", (int)st, g_fails, at_return, done);
    cudaDeviceSynchronize();
    return st == PF_ECUDA && g_fails == 1 && done == 1 ? 0 : 1;
}
