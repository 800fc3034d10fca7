// Steps of the fixed-point FP64 operators (fx.cuh) that BP3.5 (bp35_fx.cuh) and
// BP3.0 (bp30_fx.cuh) share: the factors, the chain rule at a point, and the
// derivative and transpose of a line of an element box.
#pragma once

#include "fx.cuh"

namespace fem {
namespace {

// How far (in bits) below its element's largest a node's largest line, or a
// point's largest factor, may lie.
constexpr int kFxRange = 6;

// Balanced halves of a factor scaled to 62 bits; s as in fx_magnitude.  A
// diagonal factor is positive (the element is left out otherwise).
__device__ __forceinline__ void fx_diagonal(double g, int s, int &gh, int &gl) {
    const long long m = (long long)fx_magnitude<62>(__double2hiint(g), (unsigned)__double2loint(g), s);
    gh = fx_hi(m);
    gl = fx_lo(m);
}
__device__ __forceinline__ void fx_off_diagonal(double g, int s, int &gh, int &gl) {
    const int sg = __double2hiint(g) >> 31;  // 0, or -1: negates the halves (the low one to within a unit, 2^-62)
    const long long m = (long long)fx_magnitude<62>(__double2hiint(g), (unsigned)__double2loint(g), s);
    gh = fx_hi(m) * (sg | 1);
    gl = fx_lo(m) ^ sg;
}

// (a x + b y + c z) / 2^64 of factors a, b, c below 2^62 (halves) and values
// below 2^61: the cross products are summed apart, three of them reach 2^62.6.
__device__ __forceinline__ long long fx_dot3(int ah, int al, long long x, int bh, int bl, long long y, int ch, int cl,
                                             long long z) {
    const int xh = fx_hi(x), xl = fx_lo(x), yh = fx_hi(y), yl = fx_lo(y), zh = fx_hi(z), zl = fx_lo(z);
    const long long h = mad_wide(ch, zh, mad_wide(bh, yh, mul_wide(ah, xh)));
    const long long m = mad_wide(ch, zl, mad_wide(bh, yl, mad_wide(ah, xl, 1ll << 31)));
    const long long l = mad_wide(cl, zh, mad_wide(bl, yh, mad_wide(al, xh, 1ll << 31)));
    return h + (long long)(int)(m >> 32) + (long long)(int)(l >> 32);
}

// Point l of the line of direction D at (u, v) in an element box (0: r at
// (j=u, k=v), 1: s at (i=u, k=v), 2: t at (i=u, j=v)).
template <class B, int D>
__device__ __forceinline__ int fx_at(int l, int u, int v) {
    return D == 0 ? B::at(l, u, v) : D == 1 ? B::at(u, l, v) : B::at(u, v, l);
}

// The derivatives along the lines of direction D from one box to another (or
// in place); returns the largest |high word| of the results, and in *field
// (FIELD) that of the line.
template <class B, int n, int OFF, int D, bool FIELD = false>
__device__ __forceinline__ int fx_derivative(const long long *from, long long *to, int u, int v, int *field = nullptr) {
    long long x[n];
#pragma unroll
    for (int l = 0; l < n; l++) x[l] = from[fx_at<B, D>(l, u, v)];
    if (FIELD) {
        int f = fx_line_max(x);
        if (f == 0) {  // below 2^32: tell a line of zeros from a line of small values
            int any = 0;
#pragma unroll
            for (int l = 0; l < n; l++) any |= (int)x[l];
            f = any != 0;
        }
        *field = f;
    }
    int hi = 0, lo = 0;
    fx_apply<n, n, -1, OFF>(x, [&](int l, long long y) {
        to[fx_at<B, D>(l, u, v)] = y;
        hi = max(hi, (int)(y >> 32));
        lo = min(lo, (int)(y >> 32));
    });
    return max(hi, ~lo);
}

// What fx_transpose<.., ZERO> returns for a line of zeros: more than any shift.
constexpr int kFxZeroLine = 1000;

// The transpose along a line of direction D, in place, the line first scaled
// up to QB bits; returns the shift.
template <class B, int n, int OFF, int QB, int D, bool ZERO = false>
__device__ __forceinline__ int fx_transpose(long long *box, int u, int v) {
    long long x[n];
#pragma unroll
    for (int l = 0; l < n; l++) x[l] = box[fx_at<B, D>(l, u, v)];
    const int h = max(0, QB - 32 - fx_top(fx_line_max(x)));
    if (ZERO) {
        long long any = 0;
#pragma unroll
        for (int l = 0; l < n; l++) any |= x[l];
        if (any == 0) return kFxZeroLine;
    }
#pragma unroll
    for (int l = 0; l < n; l++) x[l] <<= h;
    fx_apply<n, n, -1, OFF>(x, [&](int l, long long y) { box[fx_at<B, D>(l, u, v)] = y; });
    return h;
}

// x >> s for any s >= 0 (above 63: the sign).
__device__ __forceinline__ long long fx_shr(long long x, int s) {
    asm("shr.s64 %0, %0, %1;" : "+l"(x) : "r"(s));
    return x;
}

// Scales of an element's three directions.  With one scale for all factors, a
// flat element's small ones would keep few bits (aspect 1000: 42 of 62), and
// the result none where the derivative across the thin direction is zero.
// So where the largest diagonal factors differ by more than kFxAlike bits,
// direction d has its own scale 2^e_d, half the exponent of its largest
// diagonal factor: the factors are held as G_ab / 2^(e_a + e_b), below 1 for a
// positive definite G, and the derivatives as d_b 2^(e_b).  Elsewhere one scale
// serves.  (The kernels have a loop for each: in one, the directions' shifts
// spilled at N = 7.)
constexpr int kFxAlike = 5;
// Directions whose e_d are further apart than this leave the element to FP64:
// up to here shifting a value to another direction's scale drops no bit that
// it holds.
constexpr int kFxApart = 28;

// slot: the element's largest diagonal factors without weights (high words),
// then the largest derivatives (high words), along r, s, t.
template <int QB>
struct FxScales {
    const unsigned *slot;
    int kg;      // factors < 2^kg; split: 2 e of the direction with the largest
    int sh;      // the derivatives' common shift up
    bool split;  // a scale for each direction
    bool bad;    // out of range

    __device__ __forceinline__ int half(int d) const { return ((int)(slot[d] >> 20) - 1021) >> 1; }
    // Split: shift of direction d's line scales, and of its factors, below the largest's.
    __device__ __forceinline__ int below(int d) const { return (kg >> 1) - half(d); }
    __device__ __forceinline__ int up(int d) const { return max(0, QB - 32 - fx_top((int)slot[3 + d])); }

    __device__ __forceinline__ explicit FxScales(const unsigned *slot_) : slot(slot_) {
        const int most = __vimax3_s32((int)slot[0], (int)slot[1], (int)slot[2]),
                  least = __vimin3_s32((int)slot[0], (int)slot[1], (int)slot[2]);
        kg = (most >> 20) - 1022;
        sh = max(0, QB - 32 - fx_top(__vimax3_s32((int)slot[3], (int)slot[4], (int)slot[5])));
        split = apart(most, least);
        bad = kg > 800 || kg < -800;
        if (split) {
            const int e = (kg + 1) >> 1;
            kg = 2 * e;
            sh = __vimin3_s32(up(0) + below(0), up(1) + below(1), up(2) + below(2));
            bad = bad || e - (((least >> 20) - 1021) >> 1) > kFxApart;
        }
    }
    static __device__ __forceinline__ bool apart(int most, int least) { return (most - least) >> 20 >= kFxAlike; }
    // Whether split will be set, from the factors alone.
    static __device__ __forceinline__ bool flat(const unsigned *slot) {
        return apart(__vimax3_s32((int)slot[0], (int)slot[1], (int)slot[2]),
                     __vimin3_s32((int)slot[0], (int)slot[1], (int)slot[2]));
    }
    // All directions' below() in one word, for a later phase (fx_below).
    __device__ __forceinline__ unsigned below() const {
        return split ? (unsigned)(below(0) & 255) | (unsigned)(below(1) & 255) << 8 | (unsigned)(below(2) & 255) << 16 : 0u;
    }
    // The derivatives on one scale with their directions' 2^e, and the factors' shifts.
    __device__ __forceinline__ void scale(long long &dr, long long &ds, long long &dt, int (&s)[6]) const {
        const int a = below(0), b = below(1), c = below(2), ur = up(0), us = up(1), ut = up(2);
        dr = fx_shr(dr << ur, ur + a - sh);
        ds = fx_shr(ds << us, us + b - sh);
        dt = fx_shr(dt << ut, ut + c - sh);
        s[0] -= 2 * a;
        s[1] -= a + b;
        s[2] -= a + c;
        s[3] -= 2 * b;
        s[4] -= b + c;
        s[5] -= 2 * c;
    }
};

__device__ __forceinline__ int fx_below(unsigned word, int d) { return (int)(word >> (8 * d)) & 255; }

// What the factors of a thread's points showed: a factor above the scale
// (or not finite), a point whose diagonal factors are all far below it, a
// negative diagonal factor, and (split) the diagonal factor furthest below.
// 62 bits hold one exactly down to kFxExact bits below its scale.
constexpr int kFxExact = 9;
struct FxRange {
    int least = 0, far = 0, sign = 0, deep = 0;
    __device__ __forceinline__ bool left() const { return least < 0 || far > kFxRange || sign < 0 || deep > kFxExact; }
};

// Chain rule at a point: (wr, ws, wt) = G (dr, ds, dt) / 2^64, the factors at
// g[h plane], h = 0..5, scaled to 62 bits by eg: the scale's biased exponent
// (S.kg) with the point's weights; the derivatives as the lines left them.
template <bool SPLIT, int QB>
__device__ __forceinline__ void fx_chain(const double *g, int plane, int eg, const FxScales<QB> &S, long long dr,
                                         long long ds, long long dt, long long &wr, long long &ws, long long &wt,
                                         FxRange &range) {
    double f[6];
#pragma unroll
    for (int h = 0; h < 6; h++) f[h] = __ldg(g + h * plane);
    range.sign |= __double2hiint(f[0]) | __double2hiint(f[3]) | __double2hiint(f[5]);
    int s[6];  // (a negative diagonal factor leaves the element to FP64 whatever its s)
#pragma unroll
    for (int h = 0; h < 6; h++)
        s[h] = eg - ((h == 0 || h == 3 || h == 5) ? __double2hiint(f[h]) >> 20 : (__double2hiint(f[h]) >> 20) & 0x7ff);
    if (SPLIT) {
        S.scale(dr, ds, dt, s);
        range.deep = max(range.deep, __vimax3_s32(s[0], s[3], s[5]));
    } else {
        dr <<= S.sh;
        ds <<= S.sh;
        dt <<= S.sh;
    }
    range.least = __vimin3_s32(range.least, __vimin3_s32(s[0], s[1], s[2]), __vimin3_s32(s[3], s[4], s[5]));
    range.far = max(range.far, __vimin3_s32(s[0], s[3], s[5]));
    int h[6], l[6];
    fx_diagonal(f[0], s[0], h[0], l[0]);
    fx_off_diagonal(f[1], s[1], h[1], l[1]);
    fx_off_diagonal(f[2], s[2], h[2], l[2]);
    fx_diagonal(f[3], s[3], h[3], l[3]);
    fx_off_diagonal(f[4], s[4], h[4], l[4]);
    fx_diagonal(f[5], s[5], h[5], l[5]);
    wr = fx_dot3(h[0], l[0], dr, h[1], l[1], ds, h[2], l[2], dt);
    ws = fx_dot3(h[1], l[1], dr, h[3], l[3], ds, h[4], l[4], dt);
    wt = fx_dot3(h[2], l[2], dr, h[4], l[4], ds, h[5], l[5], dt);
}

}  // namespace
}  // namespace fem
