// Bit-sliced tiles: 32 pairs per machine word.
//
// The other filter kernels hold 32 columns of one pair in a word; shifting
// the read against the reference is then a funnel shift per plane and
// diagonal, and SneakySnake's walk a data-dependent loop whose lanes wait for
// the busiest one.  Here a word holds one column of 32 pairs (bit l = pair l
// of the group), so a diagonal is another register of the same column window
// (no shift), every decider is a fixed sequence of logic operations per column
// (no divergence), and a count is a few bit planes (a vertical counter).
// Per column, diagonal and 32 pairs: two logic operations for the mismatch
// cell (three with the reference's N folded in, which GateKeeper needs), two
// for SneakySnake, three for GateKeeper, against about 13 and 10 + a share of
// the step loop in the word-per-pair form.
//
// One warp takes a tile of G = 32 / L groups; the L lanes of a group share
// its 32 pairs and split the 2E + 1 diagonals, DPT consecutive ones per lane
// (ranges of neighbouring lanes may overlap: the ORs and ANDs over diagonals
// do not mind a diagonal taken twice).  The tile is walked in segments of
// SEG = L / 4 words, whose columns are transposed into shared memory: the
// read's in a ring that also holds the word before and the word after (the
// band reaches E < 32 columns to either side), the reference's beside it.
// The split over L lanes and the short segments keep a warp's arrays small
// (12.6 KB), so that 8 to 12 warps share an SM: the walk is a chain of
// dependent operations per column, and the loads have DRAM's latency.
//
// What bounds it: neither memory nor the integer pipe alone, but the loads'
// way through L1 (a word-wide column of pairs 20 bytes apart takes 20 sectors
// per 32 words, 9 TB/s from L2) next to the walk's latency.  At 150 bp, E = 6,
// SneakySnake alone, 4M pairs (0.29 ms), a build without the walk takes 0.19 ms,
// one without the loads 0.22 ms, one without both 0.11 ms.  Loading the words of
// a pair together (whole pairs resident: 7 warps per SM; two words per
// segment: 12.6 -> 18.7 KB) fetched two to five times fewer sectors from L2 but
// was slower (0.39 and 0.30 ms), as were separate producer and consumer warps
// per 1,024-pair tile (0.29 ms for SneakySnake, 0.42 against 0.36 ms with
// both deciders).
//
// A tile ends with the segment after which all of its pairs are decided.  The vote
// costs up to 1 % where pairs are short and some accepted (250 bp, E = 25, whole
// path: 0.697 -> 0.702 ms); 2M unrelated pairs of 300 bp at E = 8, both deciders:
// 0.46 -> 0.16 ms, 0.3M of 5,000 bp 2.0 -> 0.1.
//
// Both deciders, ms, word-per-pair kernels -> this one: 4M pairs of 150 bp at
// E = 6 0.44 -> 0.35, E = 8 0.58 -> 0.39, E = 15 1.50 -> 0.50; 2M pairs of 250 bp
// at E = 8 0.48 -> 0.34, E = 20 1.75 -> 0.52, E = 25 2.12 -> 0.56.
#pragma once
#include <climits>

#include "pf_filter.cuh"
#include "pf_kernels.h"

namespace pf {

template <int LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(r) : "r"(a), "r"(b), "r"(c), "n"(LUT));
    return r;
}

// Transpose a 32 x 32 bit matrix: bit j of a[l] becomes bit l of a[j].
__device__ __forceinline__ void transpose32(uint32_t (&a)[32]) {
#pragma unroll
    for (int l = 0; l < 16; ++l) {
        const uint32_t x = a[l], y = a[l + 16];
        a[l] = __byte_perm(x, y, 0x5410u);
        a[l + 16] = __byte_perm(x, y, 0x7632u);
    }
#pragma unroll
    for (int l = 0; l < 32; ++l) {
        if (l & 8) continue;
        const uint32_t x = a[l], y = a[l + 8];
        a[l] = __byte_perm(x, y, 0x6240u);
        a[l + 8] = __byte_perm(x, y, 0x7351u);
    }
#pragma unroll
    for (int s = 4; s >= 1; s >>= 1) {
        const uint32_t m = s == 4 ? 0x0f0f0f0fu : (s == 2 ? 0x33333333u : 0x55555555u);
#pragma unroll
        for (int l = 0; l < 32; ++l) {
            if (l & s) continue;
            const uint32_t x = a[l], y = a[l + s];
            a[l] = lop3<0xCA>(m, x, y << s);      // m ? x : y << s
            a[l + s] = lop3<0xCA>(m, x >> s, y);  // m ? x >> s : y
        }
    }
}

// Vertical counter of 32 lanes' worth of pairs: plane b[i] holds bit i of
// each pair's count, `sat` the pairs whose count passed 2^NB - 1.
template <int NB>
struct VCount {
    uint32_t b[NB];
    uint32_t sat;

    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < NB; ++i) b[i] = 0u;
        sat = 0u;
    }
    // add N bits of weight 2^LEVEL to every pair (carry-save adders)
    template <int LEVEL, int N>
    __device__ __forceinline__ void add(const uint32_t (&x)[N]) {
        if constexpr (LEVEL == NB) {
#pragma unroll
            for (int i = 0; i < N; ++i) sat |= x[i];
        } else {
            constexpr int NC = (N + 1) / 2;
            uint32_t c[NC];
            uint32_t s = b[LEVEL];
#pragma unroll
            for (int i = 0; i + 1 < N; i += 2) {
                c[i / 2] = lop3<0xE8>(s, x[i], x[i + 1]);
                s = lop3<0x96>(s, x[i], x[i + 1]);
            }
            if constexpr (N & 1) {
                c[NC - 1] = s & x[N - 1];
                s ^= x[N - 1];
            }
            b[LEVEL] = s;
            add<LEVEL + 1, NC>(c);
        }
    }
    // sum with the counter of the lane `o` away (both lanes get it)
    __device__ __forceinline__ void add_lane(int o) {
        uint32_t c = 0u;
        sat |= __shfl_xor_sync(0xffffffffu, sat, o);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const uint32_t y = __shfl_xor_sync(0xffffffffu, b[i], o);
            const uint32_t x = b[i];
            b[i] = lop3<0x96>(x, y, c);
            c = lop3<0xE8>(x, y, c);
        }
        sat |= c;
    }
    __device__ __forceinline__ void from_lane(int src) {
        sat = __shfl_sync(0xffffffffu, sat, src);
#pragma unroll
        for (int i = 0; i < NB; ++i) b[i] = __shfl_sync(0xffffffffu, b[i], src);
    }
    // the pairs whose count is past E
    __device__ __forceinline__ uint32_t above(int E) const {
        uint32_t gt = sat, eq = 0xffffffffu;
#pragma unroll
        for (int i = NB - 1; i >= 0; --i) {
            const uint32_t e = 0u - (uint32_t)((E >> i) & 1);
            gt |= eq & b[i] & ~e;
            eq &= ~(b[i] ^ e);
        }
        return gt;
    }
    // pair l's count, at most top
    __device__ __forceinline__ int get(int l, int top) const {
        int v = 0;
#pragma unroll
        for (int i = 0; i < NB; ++i) v |= (int)((b[i] >> l) & 1u) << i;
        return ((sat >> l) & 1u) ? top : imin(v, top);
    }
};

// Shape of a sliced kernel's tile: L lanes per group, DPT diagonals per lane.
template <int L, int DPT>
struct SliceShape {
    static constexpr int G = 32 / L;                 // groups per warp
    static constexpr int TILE = 32 * G;              // pairs per warp
    static constexpr int U = slice_block(L);         // columns per block
    static constexpr int SEG = slice_seg(L);         // words per segment
    static constexpr int H = L / 2;                  // lanes of each sign of d
    static constexpr int EMAX = DPT * H - 1;         // largest threshold served
    // bits of a vertical counter: exact up to EMAX, saturated beyond
    static constexpr int NB = EMAX <= 1 ? 1 : EMAX <= 3 ? 2 : EMAX <= 7 ? 3 : EMAX <= 15 ? 4 : 5;
};

// First diagonal slot (d = slot - E) of lane q of a group.  The lower half of
// the lanes covers d < 0, the upper half d >= 0 with d = 0 in slot 0 of its
// first lane (whose mismatch cells are the Hamming distance's).
template <int L, int DPT>
__device__ __forceinline__ int slice_first(int q, int E) {
    constexpr int H = L / 2;
    if constexpr (H == 1) {
        return q == 0 ? max(E - DPT, 0) : E;
    } else {
        return q < H ? max(q * (E - DPT), 0) / (H - 1) : E + ((q - H) * (E + 1 - DPT)) / (H - 1);
    }
}

// The pairs of one tile: positions [pos, pos + cnt) of a bin; pair t * 32 +
// lane of the tile is bit t * L + q of group g (lane = q * G + g), so each
// lane owns G pairs of its own group.
template <int L>
struct SlicePairs {
    static constexpr int G = 32 / L;
    int m[G];           // length; -1: absent or invalid
    unsigned invalid;   // bit t: present but its arguments are bad
    unsigned late;      // bit t: left out (leave)
    bool alone;         // for the warp to take one by one
    int mmin, mmax;     // over the tile's valid pairs (0 when there are none)
    bool full;          // all 32 * G pairs present and valid
    bool whole;         // and of one length in words

    __device__ __forceinline__ int64_t pair(const int64_t *order, int64_t pos, int t) const {
        const int64_t s = pos + 32 * t + (threadIdx.x & 31);
        return order ? __ldg(order + s) : s;
    }

    template <bool FEW>
    __device__ __forceinline__ void load(const int32_t *lens, const int16_t *Es, int E_max, int E,
                                         const int64_t *order, int64_t pos, int cnt,
                                         const LongPairs &to) {
        const int lane = threadIdx.x & 31;
        invalid = late = 0u;
        alone = false;
        int lo = INT_MAX, hi = 0;
        full = cnt == 32 * G;
#pragma unroll
        for (int t = 0; t < G; ++t) {
            m[t] = -1;
            if (32 * t + lane < cnt) {
                const int64_t p = pair(order, pos, t);
                const int len = __ldg(lens + p);
                const int e = Es ? (int)__ldg(Es + p) : E_max;
                if (len < 0 || e != E || e > E_max) {
                    invalid |= 1u << t;
                    full = false;
                } else {
                    m[t] = len;
                    lo = min(lo, len);
                    hi = max(hi, len);
                }
            }
        }
        mmin = __reduce_min_sync(0xffffffffu, lo);
        mmax = __reduce_max_sync(0xffffffffu, hi);
        const int most = 32 * (long_words(E) - 1);
        if (mmax > most) leave<FEW>(order, pos, cnt, E, most, to);
        full = __all_sync(0xffffffffu, full);
        if (mmin > mmax) mmin = mmax;  // no valid pair
        whole = full && words_of(mmin) == words_of(mmax);
    }

    // The pairs of more than `most` columns leave the tile: into the list, or, in
    // a tile of FEW (whose batch has no launch to spare), to the tile's own warp one
    // by one afterwards if they are a few among others.  FEW tiles have more than
    // four lanes per group and segments long enough for long pairs, which they walk
    // from E = 16 on faster than the word kernels.
    template <bool FEW>
    __device__ __forceinline__ void leave(const int64_t *order, int64_t pos, int cnt, int E,
                                          int most, const LongPairs &to) {
        const int lane = threadIdx.x & 31;
        bool list = to.list != nullptr, some = true;
        if (!FEW && !to.on) return;
        if (FEW || to.few) {
            int n = 0;
#pragma unroll
            for (int t = 0; t < G; ++t) n += __popc(__ballot_sync(0xffffffffu, m[t] > most));
            some = 8 * n <= cnt;
        }
        if constexpr (FEW) {
            alone = some;
            if (!alone && (E >= 16 || !list)) return;
            if (alone) list = false;
        } else if (!some) {
            return;
        }
        int lo = INT_MAX, hi = 0;
#pragma unroll
        for (int t = 0; t < G; ++t) {
            const uint32_t who = __ballot_sync(0xffffffffu, m[t] > most);
            if (who && list) {
                unsigned long long at = 0;
                if (lane == 0) at = atomicAdd(to.count, (unsigned long long)__popc(who));
                at = __shfl_sync(0xffffffffu, at, 0);
                if (m[t] > most) to.list[at + __popc(who & ((1u << lane) - 1u))] = pair(order, pos, t);
            }
            if (m[t] > most) {
                late |= 1u << t;
                m[t] = -1;
                full = false;
            } else if (m[t] >= 0) {
                lo = min(lo, m[t]);
                hi = max(hi, m[t]);
            }
        }
        mmin = __reduce_min_sync(0xffffffffu, lo);
        mmax = __reduce_max_sync(0xffffffffu, hi);
    }

    // bit of every pair of the group that has a column i
    __device__ __forceinline__ uint32_t valid(unsigned i) const {
        const int lane = threadIdx.x & 31;
        const int q = lane / G;
        uint32_t v = 0u;
#pragma unroll
        for (int t = 0; t < G; ++t) v |= ((unsigned)max(m[t], 0) > i ? 1u : 0u) << (t * L + q);
#pragma unroll
        for (int o = G; o < 32; o <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
};

// The two sides' words lie at the same offsets.
__device__ __forceinline__ bool slice_same(const PairsView &pv) {
    return pv.read.off == pv.ref.off && pv.read.stride == pv.ref.stride;
}

// The tile's columns in shared memory.  Read word w's columns lie in slot
// w % RW of the read's ring (rx: low and high code bit, rn: N), and the
// ring's first U - 1 columns a second time behind its end, so that a block
// of U columns never wraps; reference word w's in slot w % SEG (fx, fn).
template <int L>
struct SliceColumns {
    static constexpr int G = 32 / L, U = slice_block(L), SEG = slice_seg(L), RW = SEG + 2;
    static constexpr int RC = 32 * RW + U - 1, FC = 32 * SEG;   // columns
    uint2 *rx, *fx;
    uint32_t *rn, *fn;
    bool even;                  // the tile's pairs lie one stride apart
    int64_t rbase, fbase;       // even: first word of the tile's first pair,
    uint32_t rstep, fstep;      // words from a pair to the next
    int64_t *rstart, *fstart;   // else first words of the pairs, in shared memory (launches
                                // over two strided sides in pair order have none)
    int W;              // words of the tile's longest pair
    int w0, nr, nf;     // the next segment's words: first of each side, counts
    int r0;

    __device__ __forceinline__ void init(uint32_t *sm, const PairsView &pv,
                                         const SlicePairs<L> &sp, const int64_t *order,
                                         int64_t pos) {
        rx = reinterpret_cast<uint2 *>(sm);
        fx = rx + RC * G;
        rn = reinterpret_cast<uint32_t *>(fx + FC * G);
        fn = rn + RC * G;
        W = words_of(sp.mmax);
        even = true;
        if (!order && slice_strided(pv.read) && slice_strided(pv.ref)) {
            rbase = pos * pv.read.stride;
            fbase = pos * pv.ref.stride;
            rstep = (uint32_t)pv.read.stride;
            fstep = (uint32_t)pv.ref.stride;
            return;
        }
        // starts are looked up once: a pair's words are loaded in many rounds.
        // Both sides have tables here, a strided one too: where one side is not
        // even, both are loaded by them.
        const bool same = slice_same(pv);
        rstart = reinterpret_cast<int64_t *>(sm + slice_smem_words(L));
        fstart = rstart + (same ? 0 : 32 * G);
        place(pv.read, sp, order, pos, rstart, rbase, rstep);
        if (same) {
            fbase = rbase;
            fstep = rstep;
        } else {
            place(pv.ref, sp, order, pos, fstart, fbase, fstep);
        }
        even = __all_sync(0xffffffffu, even);
    }

    // Where one side's pairs lie: a table, and whether they are evenly spaced
    // (neighbours here are neighbours in memory).
    __device__ __forceinline__ void place(const SeqView &v, const SlicePairs<L> &sp,
                                          const int64_t *order, int64_t pos, int64_t *table,
                                          int64_t &base, uint32_t &step) {
        const int lane = threadIdx.x & 31;
        int64_t st[G];
#pragma unroll
        for (int t = 0; t < G; ++t) {
            st[t] = sp.m[t] > 0 ? v.start(sp.pair(order, pos, t)) : 0;
            table[32 * t + lane] = st[t];
        }
        base = __shfl_sync(0xffffffffu, st[0], 0);
        const int64_t gap = __shfl_sync(0xffffffffu, st[0], 1) - base;
        even = even && sp.whole && gap >= 0 && gap < (1 << 24);
        step = (uint32_t)gap;
#pragma unroll
        for (int t = 0; t < G; ++t) even = even && st[t] == base + (32 * t + lane) * gap;
    }

    // columns of read word w are N: before the read's start, past its end
    __device__ __forceinline__ void vacant(int w) {
        const int lane = threadIdx.x & 31;
        const int slot = (w + RW) % RW;
        uint32_t *d = rn + slot * 32 * G;
#pragma unroll
        for (int k = 0; k < G; ++k) d[k * 32 + lane] = 0xffffffffu;
        if (slot == 0)
            for (int k = lane; k < (U - 1) * G; k += 32) rn[32 * RW * G + k] = 0xffffffffu;
    }

    // The words of the segment from word w on: the read's run one ahead.
    __device__ __forceinline__ void plan(int w) {
        w0 = min(w, W);
        r0 = min(w ? w + 1 : 0, W);
        nr = min(w + SEG + 1, W) - r0;
        nf = min(w + SEG, W) - w0;
    }

    // Job j (of G lanes): one plane of one word.  Words of a plane are
    // neighbours, so that a round's loads share sectors.
    __device__ __forceinline__ void job(int j, bool &ref, int &plane, int &w) const {
        ref = j >= 3 * nr;
        const int k = ref ? j - 3 * nr : j, n = ref ? nf : nr;
        plane = k >= 2 * n ? 2 : (k >= n ? 1 : 0);
        w = (ref ? w0 : r0) + k - plane * n;
    }

    // Load the 32 words of this lane's job of the round from job j0 on.
    __device__ __forceinline__ void issue(const PairsView &pv, const SlicePairs<L> &sp,
                                          int j0, uint32_t (&x)[32]) {
        const int lane = threadIdx.x & 31;
        const int g = lane % G;
        int plane, w;
        bool ref;
        job(min(j0 + lane / G, 3 * (nr + nf) - 1), ref, plane, w);
        const SeqView &v = ref ? pv.ref : pv.read;
        const uint32_t *src = (plane == 0 ? v.lo : (plane == 1 ? v.hi : v.nm)) + w;
        const uint32_t gap = ref ? fstep : rstep;
        const uint32_t *first = src + (ref ? fbase : rbase) + (uint64_t)gap * g;
        const int64_t *st = (ref ? fstart : rstart) + g;
        const uint32_t fill = plane == 2 ? 0xffffffffu : 0u;  // past the end: N
        if (even) {
            const char *s = reinterpret_cast<const char *>(first);
            const uint32_t step = gap * (uint32_t)(G * sizeof(uint32_t));
            if (sp.whole) {
#pragma unroll
                for (int l = 0; l < 32; ++l)
                    x[l] = __ldg(reinterpret_cast<const uint32_t *>(s + (uint64_t)step * l));
                return;
            }
#pragma unroll
            for (int l = 0; l < 32; ++l) {
                const int len = __shfl_sync(0xffffffffu, sp.m[l / L], (l % L) * G + g);
                const uint32_t *y = reinterpret_cast<const uint32_t *>(s + (uint64_t)step * l);
                x[l] = len > 32 * w ? __ldg(y) : fill;
            }
        } else if (sp.whole) {
#pragma unroll
            for (int l = 0; l < 32; ++l) x[l] = __ldg(src + st[l * G]);
        } else {
#pragma unroll
            for (int l = 0; l < 32; ++l) {
                const int len = __shfl_sync(0xffffffffu, sp.m[l / L], (l % L) * G + g);
                x[l] = len > 32 * w ? __ldg(src + st[l * G]) : fill;
            }
        }
    }

    // The columns of this lane's job of the round from job j0 on.
    __device__ __forceinline__ void store(int j0, const uint32_t (&x)[32]) {
        const int lane = threadIdx.x & 31;
        const int j = j0 + lane / G;
        if (j >= 3 * (nr + nf)) return;
        int plane, w;
        bool ref;
        job(j, ref, plane, w);
        const int slot = ref ? w % SEG : w % RW;
        const int at = slot * 32 * G + lane % G;
        uint32_t *d;
        int step, wrap;
        if (plane < 2) {
            d = reinterpret_cast<uint32_t *>((ref ? fx : rx) + at) + plane;
            step = 2 * G;
            wrap = 2 * 32 * RW * G;
        } else {
            d = (ref ? fn : rn) + at;
            step = G;
            wrap = 32 * RW * G;
        }
#pragma unroll
        for (int c = 0; c < 32; ++c) d[c * step] = x[c];
        if (!ref && slot == 0) {
#pragma unroll
            for (int c = 0; c < U - 1; ++c) d[wrap + c * step] = x[c];
        }
    }

    // The columns of the segment from word w on.
    __device__ __forceinline__ void load(const PairsView &pv, const SlicePairs<L> &sp, int w) {
        plan(w);
        __syncwarp();
        for (int k = max(w ? w + 1 : 0, W); k < w + SEG + 1; ++k) vacant(k);
        const int jobs = 3 * (nr + nf);
        for (int j0 = 0; j0 < jobs; j0 += L) {
            uint32_t x[32];
            issue(pv, sp, j0, x);
            transpose32(x);
            store(j0, x);
        }
        __syncwarp();
    }
};

// AND over the group's lanes of N columns, which are counted (so it does not
// matter which lane counts which): every lane is left with N / L of them, or,
// with more lanes than columns, every L / N-th lane with one and the others
// with 0.
template <int G, int O, int N>
__device__ __forceinline__ void slice_and(uint32_t (&f)[N], uint32_t *out) {
    if constexpr (O < G) {
#pragma unroll
        for (int i = 0; i < N; ++i) out[i] = f[i];
    } else {
        const bool up = (threadIdx.x & O) != 0;
        if constexpr (N == 1) {
            uint32_t v[1] = {f[0] & __shfl_xor_sync(0xffffffffu, f[0], O)};
            slice_and<G, O / 2, 1>(v, out);
            if (up) out[0] = 0u;
        } else {
            uint32_t keep[N / 2];
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                const uint32_t send = up ? f[i] : f[N / 2 + i];
                keep[i] = (up ? f[N / 2 + i] : f[i]) & __shfl_xor_sync(0xffffffffu, send, O);
            }
            slice_and<G, O / 2, N / 2>(keep, out);
        }
    }
}

// The deciders over the columns of one tile.  D: 1 SneakySnake, 2 GateKeeper,
// 4 the Hamming count (GateKeeper needs it; with SneakySnake alone only a
// caller that resolves distances does).
//
// SneakySnake: alive[k] marks the pairs whose slot-k diagonal has met no
// obstacle since the checkpoint.  Where no lane of the group has a live
// diagonal the column is an obstacle of the snake's: counted, and every
// diagonal starts afresh at the next column (reset).
// GateKeeper: column c is amended once column c + 2 is built.
//
// SneakySnake on sub-matrices (NBY >= 0, §8.5): every diagonal starts afresh at
// a sub-matrix's first column as well, and a sub-matrix counts at most y
// obstacles: NBY bits per pair of the replications left (NBY = 0: y >= t, no
// sub-matrix has more obstacles than columns).
template <int L, int DPT, int D, int NBY = -1>
struct SliceWalk {
    using S = SliceShape<L, DPT>;
    static constexpr int G = S::G, U = S::U, NX = DPT - 1 + U;
    static constexpr bool SUB = NBY >= 0;
    static constexpr int CAP = 32 * SliceColumns<L>::RW;
    static constexpr bool SS = D & 1, GK = D & 2, HM = D & 4;

    uint2 xc[NX];                      // the lane's window of read columns
    uint32_t xn[NX];
    int pos;                           // ring column of the window's next one
    uint32_t alive[DPT], reset;
    uint32_t hist[4][GK ? DPT : 1];    // mismatch cells of the last four columns
    VCount<S::NB> ss, gk, hm;
    int t, y, tc;                      // sub-matrix columns, replications; column in it
    uint32_t left[NBY > 0 ? NBY : 1];

    __device__ __forceinline__ void clear() {
        ss.clear();
        gk.clear();
        hm.clear();
    }
    // o: the lane's first slot; the columns from read base o - E on are loaded
    __device__ __forceinline__ void init(const SliceColumns<L> &c, int o, int E) {
        const int g = (threadIdx.x & 31) % G;
        pos = o >= E ? o - E : CAP + o - E;
#pragma unroll
        for (int j = 0; j < DPT - 1; ++j) {
            xc[j] = c.rx[pos * G + g];
            xn[j] = c.rn[pos * G + g];
            pos = pos + 1 == CAP ? 0 : pos + 1;
        }
#pragma unroll
        for (int k = 0; k < DPT; ++k) alive[k] = 0u;
        reset = 0xffffffffu;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int k = 0; k < (GK ? DPT : 1); ++k) hist[j][k] = 0u;
    }

    // U columns from reference slot column f on.  v[u]: the pairs that have
    // column u; the others' cells count for nothing (GateKeeper sees them as 0).
    __device__ __forceinline__ void block(const SliceColumns<L> &c, int f, const uint32_t (&v)[U]) {
        const int g = (threadIdx.x & 31) % G;
        uint32_t m[GK ? U : 1][DPT], obs[U], ham[U];
        const uint2 *rx = c.rx + pos * G + g, *fx = c.fx + f * G + g;
        const uint32_t *rn = c.rn + pos * G + g, *fn = c.fn + f * G + g;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            xc[DPT - 1 + u] = rx[u * G];
            xn[DPT - 1 + u] = rn[u * G];
        }
        pos = pos + U >= CAP ? pos + U - CAP : pos + U;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint2 fc = fx[u * G];
            const uint32_t fnm = fn[u * G];
            uint32_t any = 0u;
            if constexpr (SUB) {
                if (tc == 0) {
                    reset = 0xffffffffu;
#pragma unroll
                    for (int i = 0; i < NBY; ++i) left[i] = (y >> i) & 1 ? 0xffffffffu : 0u;
                }
                tc = tc + 1 == t ? 0 : tc + 1;
            }
#pragma unroll
            for (int k = 0; k < DPT; ++k) {
                uint32_t t = lop3<0xBE>(xc[u + k].x, fc.x, xn[u + k]);  // (x ^ f) | n
                t = lop3<0xBE>(xc[u + k].y, fc.y, t);
                if constexpr (GK) m[u][k] = t = lop3<0xA8>(t, fnm, v[u]);  // (t | n) & v
                if constexpr (HM)
                    if (k == 0) ham[u] = GK ? t : lop3<0xA8>(t, fnm, v[u]);
                if constexpr (SS) {
                    alive[k] = lop3<0x54>(alive[k], reset, t);          // (alive | reset) & ~t
                    any |= alive[k];
                }
            }
            if constexpr (SS) {
#pragma unroll
                for (int o = G; o < 32; o <<= 1) any |= __shfl_xor_sync(0xffffffffu, any, o);
                reset = GK ? ~any & v[u] : lop3<0x8A>(any, fnm, v[u]);  // (~any | n) & v
                obs[u] = reset;
                if constexpr (NBY > 0) {
                    uint32_t some = 0u;
#pragma unroll
                    for (int i = 0; i < NBY; ++i) some |= left[i];
                    uint32_t take = obs[u] &= some;
#pragma unroll
                    for (int i = 0; i < NBY; ++i) {
                        const uint32_t b = left[i];
                        left[i] = b ^ take;
                        take &= ~b;
                    }
                }
            }
        }
        if constexpr (SS) ss.template add<0, U>(obs);
        if constexpr (HM) hm.template add<0, U>(ham);
        if constexpr (GK) {
            uint32_t a[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                a[u] = 0xffffffffu;
#pragma unroll
                for (int k = 0; k < DPT; ++k) {
                    auto col = [&](int j) { return j < 0 ? hist[4 + j][k] : m[j][k]; };
                    uint32_t t = lop3<0xE0>(col(u - 3), col(u - 1), col(u));  // l1 & (r1 | r2)
                    t = lop3<0xF8>(t, col(u - 4), col(u - 1));                // | (l2 & r1)
                    a[u] = lop3<0xE0>(a[u], t, col(u - 2));                   // & (H | t)
                }
            }
            constexpr int NC = U > L ? U / L : 1;
            uint32_t mine[NC];
            slice_and<G, 16, U>(a, mine);
            gk.template add<0, NC>(mine);
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int k = 0; k < DPT; ++k) hist[j][k] = m[U - 4 + j][k];
        }
#pragma unroll
        for (int j = 0; j < DPT - 1; ++j) {
            xc[j] = xc[j + U];
            xn[j] = xn[j + U];
        }
    }

    // Whether columns from i on can change nothing: every pair that has them
    // (GateKeeper's counts lag `extra` columns) is past E by each decider.
    __device__ __forceinline__ bool decided(const SlicePairs<L> &sp, int E, unsigned i,
                                            unsigned extra) const {
        uint32_t open = 0xffffffffu;
        if (!sp.full || i - extra >= (unsigned)sp.mmin) open = sp.valid(i - extra);
        if constexpr (SS)
            if (__any_sync(0xffffffffu, open & ~ss.above(E))) return false;
        if constexpr (GK) {
            const int g = (threadIdx.x & 31) % G;
            const uint32_t h = __shfl_sync(0xffffffffu, hm.above(E), S::H * G + g);
            if (__any_sync(0xffffffffu, open & ~h)) return false;
            VCount<S::NB> sum = gk;
#pragma unroll
            for (int x = G; x < 32; x <<= 1) sum.add_lane(x);
            if (__any_sync(0xffffffffu, open & ~sum.above(E))) return false;
        }
        return true;
    }
};

// Walk a tile's columns: positions [pos, pos + cnt) of a bin whose pairs all
// have threshold E (others are invalid), `extra` columns past the last, with
// the warp's arrays at sm.
template <int L, int DPT, typename Walk>
__device__ __forceinline__ void slice_walk(const FilterArgs &a, const SlicePairs<L> &sp,
                                           const int64_t *order, int64_t pos, int E,
                                           unsigned extra,
                                           uint32_t *sm, Walk &w) {
    using S = SliceShape<L, DPT>;
    constexpr int G = S::G, U = S::U, SEG = S::SEG;
    const int lane = threadIdx.x & 31;
    // (unsigned: columns past a length near INT_MAX)
    const unsigned total = (unsigned)sp.mmax + extra;
    const int words = (int)((total + 31u) >> 5);
    const bool one = sp.mmin == sp.mmax;
    SliceColumns<L> c;
    c.init(sm, a.pairs, sp, order, pos);
    w.clear();
    __syncwarp();
    c.vacant(-1);
    for (int w0 = 0; w0 < words; w0 += SEG) {
        const unsigned i0 = 32u * (unsigned)w0;
        c.load(a.pairs, sp, w0);
        if (w0 == 0) w.init(c, slice_first<L, DPT>(lane / G, E), E);
        const int cols = (int)min(32u * SEG, total - i0);
        for (int f = 0; f < cols; f += U) {
            uint32_t v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = 0xffffffffu;
            if (i0 + f + U > (unsigned)sp.mmin) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const unsigned i = i0 + f + u;
                    v[u] = one ? (i < (unsigned)sp.mmax ? 0xffffffffu : 0u) : sp.valid(i);
                }
            }
            w.block(c, f, v);
        }
        // (an obstacle of unrelated pairs comes every four columns or more; the
        // last words are not worth a vote)
        const unsigned i = i0 + 32u * SEG;
        if (i >= 3u * E && i + 64u <= total && w.decided(sp, E, i, extra)) break;
    }
}

// Returns the bits of the pairs that the warp has to take one by one.
template <int L, int DPT, int D, bool FEW>
__device__ __forceinline__ unsigned filter_sliced_tile(const BatchArgs &b, const int64_t *order,
                                                       int64_t pos, int cnt, int E, uint32_t *sm) {
    const FilterArgs &a = b.f;
    using S = SliceShape<L, DPT>;
    constexpr int G = S::G;
    const int lane = threadIdx.x & 31;
    const int q = lane / G, g = lane % G;
    SlicePairs<L> sp;
    sp.template load<FEW>(a.lens, a.E, a.E_max, E, order, pos, cnt, b.late);
    SliceWalk<L, DPT, D> w;
    // the last amend looks two columns ahead
    slice_walk<L, DPT>(a, sp, order, pos, E, (D & 2) ? 2 : 0, sm, w);
    if constexpr (D & 2) {
#pragma unroll
        for (int x = G; x < 32; x <<= 1) w.gk.add_lane(x);
    }
    if constexpr (D & 4) w.hm.from_lane(S::H * G + g);
#pragma unroll
    for (int t = 0; t < G; ++t) {
        if (32 * t + lane >= cnt || ((sp.late >> t) & 1u)) continue;
        const int64_t p = sp.pair(order, pos, t);
        if ((sp.invalid >> t) & 1u) {
            write_invalid<D & 3>(a, p);
            continue;
        }
        const int l = t * L + q;
        const int top = E + 1;
        const int ssc = (D & 1) ? w.ss.get(l, top) : 0;
        const int h = (D & 4) ? w.hm.get(l, top) : 0;
        int gkc = 0;
        if constexpr (D & 2) gkc = h <= E ? h : w.gk.get(l, top);
        write_outputs<D & 3>(a, p, E, ssc, gkc, h);
    }
    return sp.alone ? sp.late : 0u;
}

// SneakySnake on sub-matrices of t columns with y replications, the whole batch
// at threshold a.E_max.
template <int L, int DPT, int NBY>
__global__ void __launch_bounds__(32, slice_warps(DPT, false))
submat_sliced_kernel(FilterArgs a, int t, int y, LongPairs late) {
    extern __shared__ __align__(16) uint32_t slice_sm[];
    using S = SliceShape<L, DPT>;
    const int lane = threadIdx.x & 31;
    const int E = a.E_max;
    for (int64_t pos = (int64_t)blockIdx.x * S::TILE; pos < a.n; pos += (int64_t)gridDim.x * S::TILE) {
        const int cnt = (int)min((int64_t)S::TILE, a.n - pos);
        SlicePairs<L> sp;
        sp.template load<false>(a.lens, nullptr, E, E, nullptr, pos, cnt, late);
        SliceWalk<L, DPT, 1, NBY> w;
        w.t = t;
        w.y = y;
        w.tc = 0;
        slice_walk<L, DPT>(a, sp, nullptr, pos, E, 0, slice_sm, w);
#pragma unroll
        for (int k = 0; k < S::G; ++k) {
            if (32 * k + lane >= cnt) continue;
            const int64_t p = pos + 32 * k + lane;
            if ((sp.late >> k) & 1u) {
                if (late.few) a.count[p] = kLeftOut;
                continue;
            }
            if ((sp.invalid >> k) & 1u) write_invalid<1>(a, p);
            else write_outputs<1>(a, p, E, w.ss.get(k * L + lane / S::G, E + 1), 0, 0);
        }
    }
}

// One warp per pair: bit t of a lane's `late` is pair 32 t + lane from pos on.
template <int DEC>
__device__ __forceinline__ void slice_alone(const FilterArgs &a, const int64_t *order, int64_t pos,
                                            unsigned late) {
    const int lane = threadIdx.x & 31;
    while (__any_sync(0xffffffffu, late != 0u)) {
        const int first = late ? 32 * (__ffs(late) - 1) + lane : INT_MAX;
        const int q = __reduce_min_sync(0xffffffffu, first);
        const int64_t p = order ? __ldg(order + pos + q) : pos + q;
        filter_group<32, 2, DEC, -1>(a, p, lane, 0xffffffffu);
        if (first == q) late &= late - 1u;
    }
}

// Persistent one-warp blocks take tiles of a bin through the bin's counter.
template <int L, int DPT, int D>
__global__ void __launch_bounds__(32, slice_warps(DPT, D & 2))
filter_sliced_kernel(BatchArgs b, int bin, int E) {
    extern __shared__ __align__(16) uint32_t slice_sm[];
    if (b.layout && *b.layout != b.want) return;
    constexpr int TILE = SliceShape<L, DPT>::TILE;
    const int64_t lo = b.bin_start[bin], hi = b.bin_start[bin + 1];
    const int64_t *order = (b.order && !(b.ident && *b.ident)) ? b.order : nullptr;
    unsigned long long item = 0, next = 0;
    if (threadIdx.x == 0) item = atomicAdd(b.work + bin, 1ull);
    for (;;) {
        item = __shfl_sync(0xffffffffu, item, 0);
        const int64_t s = lo + (int64_t)item * TILE;
        if (s >= hi) break;
        if (threadIdx.x == 0) next = atomicAdd(b.work + bin, 1ull);  // known when this one is done
        const int cnt = (int)min((int64_t)TILE, hi - s);
        const unsigned late = filter_sliced_tile<L, DPT, D, (L > 4)>(b, order, s, cnt, E, slice_sm);
        if constexpr (L > 4) slice_alone<D & 3>(b.f, order, s, late);
        item = next;
    }
}

// A tile of several bins: tile t of the bins' tiles, lane i holding bin i's
// positions [lo, hi) and the tiles of bins 0..i in inc.
struct SliceBinScan {
    int64_t lo, hi, tiles, inc, total;

    template <int TILE>
    __device__ __forceinline__ void scan(const BatchArgs &b, const SliceBins &bins) {
        const int lane = threadIdx.x & 31;
        const int bin = lane < bins.count ? bins.bin[lane] : 0;
        lo = lane < bins.count ? b.bin_start[bin] : 0;
        hi = lane < bins.count ? b.bin_start[bin + 1] : 0;
        span<TILE>();
    }
    template <int TILE>
    __device__ __forceinline__ void span() {
        const int lane = threadIdx.x & 31;
        tiles = (hi - lo + TILE - 1) / TILE;
        inc = tiles;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        total = __shfl_sync(0xffffffffu, inc, 31);
    }
    template <int TILE>
    __device__ __forceinline__ int find(int64_t t, int64_t &pos, int &cnt) const {
        const int i = __popc(__ballot_sync(0xffffffffu, inc <= t));
        pos = __shfl_sync(0xffffffffu, lo + (t - (inc - tiles)) * TILE, i);
        cnt = (int)min((int64_t)TILE, __shfl_sync(0xffffffffu, hi, i) - pos);
        return i;
    }
};

// Several bins in one persistent launch: with a launch per threshold, bins
// shorter than a wave of warps (0.47M pairs) leave much of the GPU idle.  3M
// pairs in the grouped layout, both deciders: thresholds 0..25 0.94 -> 0.71 ms,
// eight thresholds up to 20 0.59 -> 0.56 ms.
template <int DPT, int D>
__global__ void __launch_bounds__(32, slice_warps(DPT, D & 2))
filter_sliced_bins_kernel(BatchArgs b, SliceBins bins) {
    extern __shared__ __align__(16) uint32_t slice_sm[];
    constexpr int TILE = SliceShape<4, DPT>::TILE;
    const int lane = threadIdx.x & 31;
    const int64_t *order = (b.order && !(b.ident && *b.ident)) ? b.order : nullptr;
    if (b.layout && *b.layout != b.want) return;
    SliceBinScan sc;
    sc.scan<TILE>(b, bins);
    unsigned long long *work = b.work + bins.bin[0];
    unsigned long long item = 0, next = 0;
    if (lane == 0) item = atomicAdd(work, 1ull);
    for (;;) {
        item = __shfl_sync(0xffffffffu, item, 0);
        if ((int64_t)item >= sc.total) break;
        if (lane == 0) next = atomicAdd(work, 1ull);
        int64_t s;
        int cnt;
        // the largest thresholds first: their tiles take longest
        const int E = bins.E[sc.find<TILE>(sc.total - 1 - (int64_t)item, s, cnt)];
        filter_sliced_tile<4, DPT, D, false>(b, order, s, cnt, E, slice_sm);
        item = next;
    }
}

// L lanes per group with L > 4: fewer pairs per warp and longer segments (L / 4
// words).  For batches too small to fill the GPU with tiles of many groups,
// where a tile's latency and not the rate counts, and for pairs whose words are
// scattered over the planes: a segment's words of a pair share sectors.
// One launch over all tiles of the bins, or, with single >= 0, over the whole
// batch at that threshold.
template <int L, int D>
__global__ void __launch_bounds__(32, L == 8 ? 8 : 12)
filter_sliced_small_kernel(BatchArgs b, SliceBins bins, int single) {
    extern __shared__ __align__(16) uint32_t slice_sm[];
    constexpr int TILE = 32 * (32 / L);
    if (b.layout && *b.layout != b.want) return;
    SliceBinScan sc;
    if (single < 0) {
        sc.scan<TILE>(b, bins);
    } else {
        sc.lo = 0;
        sc.hi = (threadIdx.x & 31) == 0 ? b.f.n : 0;
        sc.span<TILE>();
    }
    const int64_t *order = (b.order && !(b.ident && *b.ident)) ? b.order : nullptr;
    // the largest thresholds first: their tiles take longest
    for (int64_t t = sc.total - 1 - (int64_t)blockIdx.x; t >= 0; t -= gridDim.x) {
        int64_t s;
        int cnt;
        const int i = sc.find<TILE>(t, s, cnt);
        const int E = single < 0 ? bins.E[i] : single;
        // diagonals per lane: those of the largest threshold of E's class
        constexpr int H = L / 2;
        unsigned late = 0u;
        switch (E >> 3) {
            case 0:  // (eight lanes take single thresholds from 8 on only)
                if constexpr (L > 8)
                    late = filter_sliced_tile<L, (7 + H) / H, D, true>(b, order, s, cnt, E, slice_sm);
                break;
            case 1: late = filter_sliced_tile<L, (15 + H) / H, D, true>(b, order, s, cnt, E, slice_sm); break;
            case 2: late = filter_sliced_tile<L, (23 + H) / H, D, true>(b, order, s, cnt, E, slice_sm); break;
            default: late = filter_sliced_tile<L, (31 + H) / H, D, true>(b, order, s, cnt, E, slice_sm); break;
        }
        slice_alone<D & 3>(b.f, order, s, late);
    }
}

}  // namespace pf
