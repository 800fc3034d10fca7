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

// The transpose along a line of direction D, in place, the line first scaled
// up to QB bits; returns the shift.
template <class B, int n, int OFF, int QB, int D>
__device__ __forceinline__ int fx_transpose(long long *box, int u, int v) {
    long long x[n];
#pragma unroll
    for (int l = 0; l < n; l++) x[l] = box[fx_at<B, D>(l, u, v)];
    const int h = max(0, QB - 32 - fx_top(fx_line_max(x)));
#pragma unroll
    for (int l = 0; l < n; l++) x[l] <<= h;
    fx_apply<n, n, -1, OFF>(x, [&](int l, long long y) { box[fx_at<B, D>(l, u, v)] = y; });
    return h;
}

// What the factors of a thread's points showed: a factor above the element's
// largest diagonal one (or not finite), a point whose diagonal factors are
// all far below it, a negative diagonal factor.
struct FxRange {
    int least = 0, far = 0, sign = 0;
    __device__ __forceinline__ bool left() const { return least < 0 || far > kFxRange || sign < 0; }
};

// Chain rule at a point: (wr, ws, wt) = G (dr, ds, dt) / 2^64, the factors at
// g[h plane], h = 0..5, scaled to 62 bits by eg: the largest diagonal factor's
// biased exponent with the point's weights.
__device__ __forceinline__ void fx_chain(const double *g, int plane, int eg, long long dr, long long ds, long long dt,
                                         long long &wr, long long &ws, long long &wt, FxRange &range) {
    double f[6];
#pragma unroll
    for (int h = 0; h < 6; h++) f[h] = __ldg(g + h * plane);
    range.sign |= __double2hiint(f[0]) | __double2hiint(f[3]) | __double2hiint(f[5]);
    const int s0 = eg - (__double2hiint(f[0]) >> 20), s3 = eg - (__double2hiint(f[3]) >> 20),
              s5 = eg - (__double2hiint(f[5]) >> 20), s1 = eg - ((__double2hiint(f[1]) >> 20) & 0x7ff),
              s2 = eg - ((__double2hiint(f[2]) >> 20) & 0x7ff), s4 = eg - ((__double2hiint(f[4]) >> 20) & 0x7ff);
    range.least = __vimin3_s32(range.least, __vimin3_s32(s0, s1, s2), __vimin3_s32(s3, s4, s5));
    range.far = max(range.far, __vimin3_s32(s0, s3, s5));
    int h[6], l[6];
    fx_diagonal(f[0], s0, h[0], l[0]);
    fx_off_diagonal(f[1], s1, h[1], l[1]);
    fx_off_diagonal(f[2], s2, h[2], l[2]);
    fx_diagonal(f[3], s3, h[3], l[3]);
    fx_off_diagonal(f[4], s4, h[4], l[4]);
    fx_diagonal(f[5], s5, h[5], l[5]);
    wr = fx_dot3(h[0], l[0], dr, h[1], l[1], ds, h[2], l[2], dt);
    ws = fx_dot3(h[1], l[1], dr, h[3], l[3], ds, h[4], l[4], dt);
    wt = fx_dot3(h[2], l[2], dr, h[4], l[4], ds, h[5], l[5], dt);
}

}  // namespace
}  // namespace fem
