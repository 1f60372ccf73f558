// a6: verification device function, dist = min(Levenshtein(read, ref), E + 1), exact.
//
// The thesis verifies the mappings that pass the filter with banded
// Levenshtein distance (Ch. 2, "Accelerating Read Alignment": Ukkonen's
// band of 2E+1 diagonals).  This kernel computes that band with bit
// vectors: one machine word holds the vertical differences of the 2E+1
// band cells of a DP column (Myers 1999; Hyyrö 2003), one thread per pair (or
// two pairs, further down).
//
// Rows are read prefixes (row i = read[0..i)), columns reference prefixes.
// Column j keeps the cells of rows j-E .. j+E as
//     T  = D(j-E, j)                   (value of the top band cell)
//     VP, VN bits q-1 = +1 / -1 difference D(j-E+q) - D(j-E+q-1), q=1..2E.
// Rows above row 0 are virtual with D(i, j) = j - i, which extends the
// global boundary D(0, j) = j, D(i, 0) = i upwards; they never match.
// Step j-1 -> j runs one Myers column over rows j-E .. j+E:
//   - the vertical differences of rows j-E .. j+E-1 are those stored for
//     column j-1; row j+E (outside column j-1's band) is taken as +1,
//   - the horizontal difference entering above row j-E is taken as +1.
// Both stand-ins are upper bounds of the true values, and every DP value
// computed from upper bounds is itself an upper bound; a cell whose true
// value is <= E has an optimal path inside the band, so min(result, E+1)
// is exact.  After the column, the top row's difference updates T and the
// vectors shift down by one row.
// dist = D(m, m) = T + (sum of the first E differences) at column m.
#pragma once
#include "pf_internal.cuh"

namespace pf {

template <typename U>
struct Bits;
template <>
struct Bits<uint32_t> {
    static __device__ __forceinline__ int popc(uint32_t x) { return __popc(x); }
};
template <>
struct Bits<uint64_t> {
    static __device__ __forceinline__ int popc(uint64_t x) { return __popcll(x); }
};

// 0 or ~0: bit t of x, spread over the word.
__device__ __forceinline__ uint32_t bcast(uint32_t x, int t) {
    return (uint32_t)((int32_t)(x << (31 - t)) >> 31);
}

template <typename U>
__device__ __forceinline__ U spread(uint32_t b) {
    if constexpr (sizeof(U) == 4) return b;
    else return ((uint64_t)b << 32) | b;
}

// The read's three planes from bit 32*fw - E on: x0 covers the first 32
// bits, x1 the next 32, x2 the 32 after (used by 64-bit bands only).
struct ReadWin {
    uint32_t lo0, lo1, lo2, hi0, hi1, hi2, nm0, nm1, nm2;
};

// Bits [t, t + |U|) of the window.
template <typename U>
__device__ __forceinline__ U win(uint32_t x0, uint32_t x1, uint32_t x2, int t) {
    if constexpr (sizeof(U) == 4) {
        return __funnelshift_r(x0, x1, (unsigned)t);
    } else {
        return ((uint64_t)__funnelshift_r(x1, x2, (unsigned)t) << 32) |
               __funnelshift_r(x0, x1, (unsigned)t);
    }
}

// One DP column: reference base at bit t of the reference word f, band rows
// read from the window at offset t.  VP keeps the bottom stand-in bit set.
//
// The column's horizontal differences would enter the next row up (shift
// left, +1 entering above the top row) and the new vertical differences
// would then move down one row with the band (shift right); the two shifts
// cancel except on D0, so the new vectors come from D0 >> 1 directly.  The
// top row's new vertical difference is then never +1 and is -1 exactly when
// bit 0 of D0 is set: T grows by 1 per column, less the number of those
// bits, which go to the top of accM.
template <typename U>
__device__ __forceinline__ void column(const ReadWin &r, const Word3 &f, int t, U store_mask,
                                       U bottom, U &VP, U &VN, uint32_t &accM) {
    const U mlo = spread<U>(bcast(f.lo, t));
    const U mhi = spread<U>(bcast(f.hi, t));
    const U fn = spread<U>(bcast(f.nm, t));
    const U wlo = win<U>(r.lo0, r.lo1, r.lo2, t);
    const U whi = win<U>(r.hi0, r.hi1, r.hi2, t);
    const U wnm = win<U>(r.nm0, r.nm1, r.nm2, t);
    // Eq bit q: read base of row j-E+q equals the reference base, neither N.
    // Bits above the band (q > 2E) only ever influence higher bits (carries
    // and the left shifts run upwards), and the stored vectors drop them.
    const U Eq = ~((wlo ^ mlo) | (whi ^ mhi) | wnm | fn);
    const U X = Eq | VN;
    const U D0 = (((X & VP) + VP) ^ VP) | X;
    const U Ph = VN | ~(D0 | VP);
    const U Mh = VP & D0;
    const U D1 = D0 >> 1;
    accM = __funnelshift_r(accM, (uint32_t)D0, 1);
    VP = ((Mh | ~(D1 | Ph)) & store_mask) | bottom;
    VN = Ph & D1 & store_mask;
}

template <typename U, typename L = LdNC>
__device__ __forceinline__ int verify_pair(const PairsView &pv, int64_t p, int m, int E) {
    if (m == 0) return 0;
    const int W = (m + 31) >> 5;
    const int64_t rb = pv.read.template start<L>(p), fb = pv.ref.template start<L>(p);
    const U store_mask = (U(1) << (2 * E)) - 1;     // 2E stored differences
    const U bottom = U(1) << (2 * E);               // +1 stand-in of row j+E

    // column 0: rows -E..E hold |i|; differences -1 for rows -E+1..0,
    // +1 for rows 1..E
    U VN = (U(1) << E) - 1;
    U VP = (store_mask & ~VN) | bottom;
    int T = E;

    // Reference word fw holds columns j = 32 fw + 1 + t (t = 0..31), whose
    // band starts at read bit s = j - E - 1 = 32 fw - E + t.  Read words
    // fw-1 .. fw+2 cover every window of the word.
    const unsigned rs = 32u - (unsigned)E;
    Word3 ra = load_word<L>(pv.read, rb, -1, W);
    Word3 rb0 = load_word<L>(pv.read, rb, 0, W);
    Word3 rc = load_word<L>(pv.read, rb, 1, W);
    Word3 rd;
    if constexpr (sizeof(U) == 8) rd = load_word<L>(pv.read, rb, 2, W);
    for (int fw = 0; fw < W; ++fw) {
        const Word3 f = load_word<L>(pv.ref, fb, fw, W);
        ReadWin r;
        r.lo0 = __funnelshift_rc(ra.lo, rb0.lo, rs);
        r.hi0 = __funnelshift_rc(ra.hi, rb0.hi, rs);
        r.nm0 = __funnelshift_rc(ra.nm, rb0.nm, rs);
        r.lo1 = __funnelshift_rc(rb0.lo, rc.lo, rs);
        r.hi1 = __funnelshift_rc(rb0.hi, rc.hi, rs);
        r.nm1 = __funnelshift_rc(rb0.nm, rc.nm, rs);
        if constexpr (sizeof(U) == 8) {
            r.lo2 = __funnelshift_rc(rc.lo, rd.lo, rs);
            r.hi2 = __funnelshift_rc(rc.hi, rd.hi, rs);
            r.nm2 = __funnelshift_rc(rc.nm, rd.nm, rs);
        } else {
            r.lo2 = r.hi2 = r.nm2 = 0u;
        }
        const int ncol = min(32, m - 32 * fw);
        uint32_t accM = 0u;
        if (ncol == 32) {
#pragma unroll
            for (int t = 0; t < 32; ++t)
                column<U>(r, f, t, store_mask, bottom, VP, VN, accM);
        } else {
            for (int t = 0; t < ncol; ++t)
                column<U>(r, f, t, store_mask, bottom, VP, VN, accM);
        }
        // top cell D(j-E, j) after the word: each column adds 1 + its top
        // row's new difference (0 or -1)
        T += ncol - __popc(accM);
        // Early exit: the band's smallest value is at least T minus the
        // number of -1 differences.  Past E, every path through this column
        // costs more than E, so the distance saturates (the values that the
        // band computes are exact wherever they are <= E).
        if (T - Bits<U>::popc(VN) > E) return E + 1;
        ra = rb0;
        rb0 = rc;
        if constexpr (sizeof(U) == 8) {
            rc = rd;
            rd = load_word<L>(pv.read, rb, fw + 3, W);
        } else {
            rc = load_word<L>(pv.read, rb, fw + 2, W);
        }
    }
    const U first = (U(1) << E) - 1;
    const int dist = T + Bits<U>::popc(VP & first) - Bits<U>::popc(VN & first);
    return min(dist, E + 1);
}

// Two pairs in the halves of a word, for bands of at most 15 cells (kTwoE = 7):
// cell q of either band is bit q of its half.  The one carry of a column,
// (X & VP) + VP, has 15-bit operands and stays in its half; what the shifts
// move across the border lands above the low band, where bits only influence
// higher ones and are dropped.  Smaller thresholds share the band: the values
// up to E are the same.
//
// Both pairs run the same columns: behind its end a pair's read and reference
// continue with the same base, which leaves the distance as it is (a common
// suffix costs nothing), so lengths may differ and columns come in eights.
//
// The verifier is bound by the integer pipe; a column of two pairs takes about
// 24 instructions, of one pair 22.  2M pairs of 150 bp, E = 6: 331 us one by
// one, 234 so (more warps an SM change nothing).
constexpr int kTwoE = 7;

struct TwoPlanes {
    uint32_t z[4];   // half words 2 fw - 1 .. 2 fw + 2 of both pairs

    // The halves' bits from column T's band on: 16 bits for odd T, 15 for even.
    // (Odd columns start at even bits, so that one window in eight is a half
    // word as it stands and one a byte permutation.)
    template <int T>
    __device__ __forceinline__ uint32_t win() const {
        constexpr int S = ((T + 1) & ~1) - 1 - kTwoE + 16;
        constexpr int H = S >> 4, OFF = S & 15;
        constexpr uint32_t M = (0xffffu >> OFF) * 0x00010001u;
        uint32_t w;
        if constexpr (OFF == 0) w = z[H];
        else if constexpr (OFF == 8) w = __byte_perm(z[H], z[H + 1], 0x6341u);
        else w = ((z[H] >> OFF) & M) | ((z[H + 1] << (16 - OFF)) & ~M);
        return w >> ((T + 1) & 1);
    }
};

// 0 or 0xffff per half: bit T % 16 of each half of x.
template <int T>
__device__ __forceinline__ uint32_t bcast2(uint32_t x) {
    // the sign of byte 0 or 1 of each half, in both of its bytes; columns eight
    // apart share the shift
    const uint32_t y = x << (7 - (T & 7));
    // (asm: __byte_perm has no sign selectors)
    uint32_t r;
    asm("prmt.b32 %0, %1, 0, %2;" : "=r"(r) : "r"(y), "n"((T & 8) ? 0xbb99 : 0xaa88));
    return r;
}

struct TwoBands {
    static constexpr uint32_t kStore = ((1u << (2 * kTwoE)) - 1) * 0x00010001u;
    static constexpr uint32_t kBottom = (1u << (2 * kTwoE)) * 0x00010001u;
    TwoPlanes lo, hi, nm;
    uint32_t flo[2], fhi[2], fnm[2];   // the reference's half words
    uint32_t VP, VN;
    // columns whose D0 has bit 0 set: even columns of the low half, odd ones,
    // even of the high half, odd (a byte each, 32 columns at most)
    uint32_t top;

    template <int T>
    __device__ __forceinline__ uint32_t column() {
        constexpr int F = T >> 4;
        const uint32_t mlo = bcast2<T>(flo[F]), mhi = bcast2<T>(fhi[F]), fn = bcast2<T>(fnm[F]);
        const uint32_t t = (lo.win<T>() ^ mlo) | nm.win<T>();
        const uint32_t ne = (hi.win<T>() ^ mhi) | t;
        const uint32_t X = ~(ne | fn) | VN;
        const uint32_t D0 = (((X & VP) + VP) ^ VP) | X;
        const uint32_t Ph = VN | ~(D0 | VP);
        const uint32_t Mh = VP & D0;
        const uint32_t D1 = D0 >> 1;
        VP = ((Mh | ~(D1 | Ph)) & kStore) | kBottom;
        VN = Ph & D1 & kStore;
        return D0;
    }
    template <int T>
    __device__ __forceinline__ void two() {
        const uint32_t even = column<T>(), odd = column<T + 1>();
        top += __byte_perm(even, odd, 0x6240u) & 0x01010101u;
    }
    template <int T>
    __device__ __forceinline__ void eight() {
        two<T>();
        two<T + 2>();
        two<T + 4>();
        two<T + 6>();
    }
};

// Word w of a pair's planes, 0 (no N) behind the `rest` columns from there on.
__device__ __forceinline__ Word3 load_ended(const SeqView &s, int64_t start, int w, int W,
                                            int rest) {
    Word3 x = load_word(s, start, w, W);
    const uint32_t past = __funnelshift_lc(0u, 0xffffffffu, (unsigned)max(rest, 0));
    x.lo &= ~past;
    x.hi &= ~past;
    x.nm &= ~past;
    return x;
}

// Distances of pairs p and p2 (lengths m and m2 >= 0, thresholds at most kTwoE).
__device__ __forceinline__ void verify_two(const PairsView &pv, int64_t p, int64_t p2, int m,
                                           int m2, int E, int E2, int &dist, int &dist2) {
    const int W = words_of(m), W2 = words_of(m2);
    const int64_t ra = pv.read.start(p), rb = pv.read.start(p2);
    const int64_t fa = pv.ref.start(p), fb = pv.ref.start(p2);
    TwoBands b;
    b.VN = ((1u << kTwoE) - 1) * 0x00010001u;
    b.VP = (TwoBands::kStore & ~b.VN) | TwoBands::kBottom;
    b.top = 0u;
    auto low = [](uint32_t x, uint32_t y) { return __byte_perm(x, y, 0x5410u); };
    auto high = [](uint32_t x, uint32_t y) { return __byte_perm(x, y, 0x7632u); };
    Word3 a1 = load_ended(pv.read, ra, 0, W, m), b1 = load_ended(pv.read, rb, 0, W2, m2);
    b.lo.z[2] = b.hi.z[2] = 0u;
    b.nm.z[2] = 0xffffffffu;   // before the read nothing matches
    b.lo.z[3] = low(a1.lo, b1.lo);
    b.hi.z[3] = low(a1.hi, b1.hi);
    b.nm.z[3] = low(a1.nm, b1.nm);
    int T = kTwoE, T2 = kTwoE;
    const int words = max(W, W2);
    for (int fw = 0; fw < words; ++fw) {
        const int rest = m - 32 * fw, rest2 = m2 - 32 * fw;
        const Word3 f = load_ended(pv.ref, fa, fw, W, rest);
        const Word3 g = load_ended(pv.ref, fb, fw, W2, rest2);
        const Word3 a2 = load_ended(pv.read, ra, fw + 1, W, rest - 32);
        const Word3 b2 = load_ended(pv.read, rb, fw + 1, W2, rest2 - 32);
        auto roll = [&](TwoPlanes &x, uint32_t a_now, uint32_t b_now, uint32_t a_next,
                        uint32_t b_next) {
            x.z[0] = x.z[2];
            x.z[1] = x.z[3];
            x.z[2] = high(a_now, b_now);
            x.z[3] = low(a_next, b_next);
        };
        roll(b.lo, a1.lo, b1.lo, a2.lo, b2.lo);
        roll(b.hi, a1.hi, b1.hi, a2.hi, b2.hi);
        roll(b.nm, a1.nm, b1.nm, a2.nm, b2.nm);
        b.flo[0] = low(f.lo, g.lo);
        b.flo[1] = high(f.lo, g.lo);
        b.fhi[0] = low(f.hi, g.hi);
        b.fhi[1] = high(f.hi, g.hi);
        b.fnm[0] = low(f.nm, g.nm);
        b.fnm[1] = high(f.nm, g.nm);
        const int left = min(max(rest, rest2), 32);
        b.eight<0>();
        if (left > 8) b.eight<8>();
        if (left > 16) b.eight<16>();
        if (left > 24) b.eight<24>();
        // as in verify_pair: out when both pairs are over, by their bands'
        // smallest values past the thresholds or by their ends (the columns
        // behind a pair's end leave its distance as it is, so a short pair or an
        // absent one does not hold a long one)
        const int ran = (left + 7) & ~7;
        T += ran - (int)((b.top & 0xffu) + ((b.top >> 8) & 0xffu));
        T2 += ran - (int)(((b.top >> 16) & 0xffu) + (b.top >> 24));
        b.top = 0u;
        if ((rest <= 32 || T - __popc(b.VN & 0xffffu) > E) &&
            (rest2 <= 32 || T2 - __popc(b.VN >> 16) > E2))
            break;
        a1 = a2;
        b1 = b2;
    }
    constexpr uint32_t first = (1u << kTwoE) - 1;
    dist = min(T + __popc(b.VP & first) - __popc(b.VN & first), E + 1);
    dist2 = min(T2 + __popc((b.VP >> 16) & first) - __popc((b.VN >> 16) & first), E2 + 1);
}

}  // namespace pf
