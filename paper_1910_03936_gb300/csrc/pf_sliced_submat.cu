// SneakySnake on sub-matrices with bit-sliced tiles (pf_sliced.cuh).
#include <algorithm>

#include "pf_sliced.cuh"

namespace pf {

namespace {

template <int L, int DPT, int NBY>
cudaError_t go(const FilterArgs &a, int t, int y, const LongPairs &late, int sms, cudaStream_t st) {
    BatchArgs b{};
    b.f = a;
    const int64_t tiles = (a.n + SliceShape<L, DPT>::TILE - 1) / SliceShape<L, DPT>::TILE;
    const int64_t grid = std::min<int64_t>(tiles, (int64_t)sms * slice_warps(DPT, false));
    submat_sliced_kernel<L, DPT, NBY>
        <<<(unsigned)grid, 32, slice_smem_bytes(L, b), st>>>(a, t, y, late);
    return cudaGetLastError();
}

template <int L, int DPT>
cudaError_t by_y(const FilterArgs &a, int t, int y, const LongPairs &late, int sms, cudaStream_t st) {
    if (y >= t) return go<L, DPT, 0>(a, t, y, late, sms, st);
    if (y <= 3) return go<L, DPT, 2>(a, t, y, late, sms, st);
    return go<L, DPT, 5>(a, t, y, late, sms, st);
}

}  // namespace

cudaError_t launch_submat_sliced(const FilterArgs &a, int t, int y, int lanes, const LongPairs &late,
                                 int sms, cudaStream_t st) {
    const int E = a.E_max;
    if (lanes == 16) {
        if (E <= 15) return by_y<16, 2>(a, t, y, late, sms, st);
        if (E <= 23) return by_y<16, 3>(a, t, y, late, sms, st);
        return by_y<16, 4>(a, t, y, late, sms, st);
    }
    if (E <= 1) return by_y<4, 1>(a, t, y, late, sms, st);
    if (E <= 3) return by_y<4, 2>(a, t, y, late, sms, st);
    if (E <= 5) return by_y<4, 3>(a, t, y, late, sms, st);
    if (E <= 7) return by_y<4, 4>(a, t, y, late, sms, st);
    if (E <= 11) return by_y<4, 6>(a, t, y, late, sms, st);
    if (E <= 15) return by_y<4, 8>(a, t, y, late, sms, st);
    if (E <= 25) return by_y<4, 13>(a, t, y, late, sms, st);
    return by_y<4, 16>(a, t, y, late, sms, st);
}

}  // namespace pf
