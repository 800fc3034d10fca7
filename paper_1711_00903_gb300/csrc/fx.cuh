// One-dimensional contractions of FP64 data on the integer multiply-add
// pipe: exact 64-bit fixed point in place of FP64 arithmetic.
//
// GB300 issues 2 FP64 FMAs per clock per SM and 32 of the 32 x 32 + 64 bit
// integer multiply-adds (measured: 1.7 against 29).  A line of an element is
// therefore contracted on 64-bit integers: values x (|x| < 2^61) and operator
// entries C (scaled to 64 bits, rounded once on the host) are split into
// balanced 32-bit halves,
//   x = xh 2^32 + xl,  C = Ch 2^32 + Cl,  -2^31 <= xl, Cl < 2^31,
// and y = sum C x / 2^64 is accumulated as sum Ch xh + (sum Ch xl + Cl xh) /
// 2^32: three integer multiply-adds per term, exact up to the last unit (the
// product Cl xl, under a quarter of a unit, is dropped).  A value carries 60
// to 61 bits against FP64's 53, so a line's rounding error is below that of
// the FP64 line as long as the line's values share a scale; the kernels
// choose the scales (bp35_fx.cuh) and fall back to FP64 where an element's
// values do not share one.  A line of 8 values costs 0.4 clocks per value and
// SM this way against 3.1 on the FP64 pipe.
//
// The multiply-add is written as mad.lo.cc / madc.hi, which compiles to one
// instruction; mad.wide.s32, or a 64-bit product and sum in C, compiles to a
// product and a separate 64-bit addition and measured a quarter slower (n =
// 8, both with the addition on the otherwise idle integer pipe).
//
// The operators are the even-odd folded ones of eo.cuh.  The transposed
// ones also carry the quadrature weights' powers of two, A'[i][l] =
// A[i][l] 2^(w_l - w_i) (w_l: exponent of the weight of point l), so that a
// line of values that each hold a quadrature weight (the factors do) is
// stored without it: otherwise the small weights at an element's edges
// would cost its edge nodes their leading bits (4 bits a direction at
// N = 15).  Powers of two keep everything exact.
#pragma once

#include "eo.cuh"
#include "fx_layout.h"

namespace fem {

static __constant__ FxEntry c_fx[kFoldTotal];
static __constant__ FxDegree c_fxd[kMaxN + 1];

// a b, and a b + c, of signed 32-bit factors in 64 bits.
__device__ __forceinline__ long long mul_wide(int a, int b) {
    long long d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
}
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
    int lo, hi;
    asm("mad.lo.cc.s32 %0, %2, %3, %4;\n madc.hi.s32 %1, %2, %3, %5;"
        : "=&r"(lo), "=r"(hi)
        : "r"(a), "r"(b), "r"((int)c), "r"((int)(c >> 32)));
    return ((long long)hi << 32) | (unsigned)lo;
}

// Balanced halves of a 64-bit integer.
__device__ __forceinline__ int fx_lo(long long x) { return (int)x; }
__device__ __forceinline__ int fx_hi(long long x) { return (int)(x >> 32) + (int)((unsigned)x >> 31); }

// Sum of products of one output: h of the high halves, m the cross products.
struct FxSum {
    long long h, m;
    __device__ __forceinline__ void set(int ch, int cl, int xh, int xl) {
        h = mul_wide(ch, xh);
        m = mad_wide(cl, xh, mad_wide(ch, xl, 1ll << 31));  // halved to nearest
    }
    __device__ __forceinline__ void add(int ch, int cl, int xh, int xl) {
        h = mad_wide(ch, xh, h);
        m = mad_wide(ch, xl, m);
        m = mad_wide(cl, xh, m);
    }
    __device__ __forceinline__ long long value() const { return h + (long long)(int)(m >> 32); }
};

// y (P) = A x (Q) along one line, A folded at table offset OFF with parity
// SIG (eo.cuh), scaled by 2^-tau (FxDegree): |y| < 1.02 2^B for |x| < 2^B, B =
// fx_bits35, kFxBits30.  put(a, y_a) takes each output as it is formed, so
// that a line needs the registers of its folded inputs and two sums only.
template <int P, int Q, int SIG, int OFF, class F>
__device__ __forceinline__ void fx_apply(const long long (&x)[Q], F &&put) {
    constexpr int hp = P / 2, hq = Q / 2;
    constexpr int oS = OFF, oT = OFF + hp * hq, oC = OFF + 2 * hp * hq;
    constexpr int oR = oC + ((Q % 2) ? hp : 0);
    static_assert(Q >= 2, "lines have at least two points");
    int eh[hq], el[hq], oh[hq], ol[hq];
#pragma unroll
    for (int i = 0; i < hq; i++) {
        const long long e = x[i] + x[Q - 1 - i], o = x[i] - x[Q - 1 - i];
        eh[i] = fx_hi(e);
        el[i] = fx_lo(e);
        oh[i] = fx_hi(o);
        ol[i] = fx_lo(o);
    }
    int mh = 0, ml = 0;  // the middle value, doubled (its table entries are halved)
    if (Q % 2) {
        const long long d = x[hq] + x[hq];
        mh = fx_hi(d);
        ml = fx_lo(d);
    }
#pragma unroll
    for (int a = 0; a < hp; a++) {
        FxSum E, O;
        E.set(c_fx[oS + a * hq].h, c_fx[oS + a * hq].l, eh[0], el[0]);
        O.set(c_fx[oT + a * hq].h, c_fx[oT + a * hq].l, oh[0], ol[0]);
#pragma unroll
        for (int i = 1; i < hq; i++) {
            E.add(c_fx[oS + a * hq + i].h, c_fx[oS + a * hq + i].l, eh[i], el[i]);
            O.add(c_fx[oT + a * hq + i].h, c_fx[oT + a * hq + i].l, oh[i], ol[i]);
        }
        if (Q % 2) E.add(c_fx[oC + a].h, c_fx[oC + a].l, mh, ml);
        const long long ve = E.value(), vo = O.value();
        put(a, ve + vo);
        put(P - 1 - a, (SIG > 0) ? (ve - vo) : (vo - ve));
    }
    if (P % 2) {
        FxSum M;
        M.set(c_fx[oR].h, c_fx[oR].l, (SIG > 0) ? eh[0] : oh[0], (SIG > 0) ? el[0] : ol[0]);
#pragma unroll
        for (int i = 1; i < hq; i++)
            M.add(c_fx[oR + i].h, c_fx[oR + i].l, (SIG > 0) ? eh[i] : oh[i], (SIG > 0) ? el[i] : ol[i]);
        if ((Q % 2) && SIG > 0) M.add(c_fx[oR + hq].h, c_fx[oR + hq].l, mh, ml);
        put(hp, M.value());
    }
}

// High word of |d| (monotone in |d|, the exponent in its top 11 bits).
__device__ __forceinline__ int fx_abs_hi(double d) { return __double2hiint(d) & 0x7fffffff; }

// |g| 2^(bits - k) as an integer below 2^bits, given s = (largest biased
// exponent, that of 2^(k-1)) - (biased exponent of g) >= 0; truncated.
// hi, lo: the words of g.
template <int bits>
__device__ __forceinline__ unsigned long long fx_magnitude(int hi, unsigned lo, int s) {
    const unsigned mh = __funnelshift_l(lo, ((unsigned)hi & 0xfffffu) | 0x100000u, bits - 53);
    unsigned long long m = ((unsigned long long)mh << 32) | (lo << (bits - 53));
    asm("shr.u64 %0, %0, %1;" : "+l"(m) : "r"(s));  // s above 63 gives 0 (zeros, tiny values)
    return m;
}

// g 2^(bits - k), signed.
template <int bits>
__device__ __forceinline__ long long fx_from_double(double g, int s) {
    const int hi = __double2hiint(g);
    const long long sg = (long long)(hi >> 31);
    return ((long long)fx_magnitude<bits>(hi, (unsigned)__double2loint(g), s) ^ sg) - sg;
}

// (double)x 2^k, |k| < 960.
__device__ __forceinline__ double fx_to_double(long long x, int k) {
    const double d = __ll2double_rn(x);
    return x == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + k * (1 << 20), __double2loint(d));
}

// Bit length of a non-negative word: x < 2^(32 + fx_top(h)) for the high
// word h of x.
__device__ __forceinline__ int fx_top(int h) { return 32 - __clz(h); }

// Largest |high word| of the values of a line (of ~h for negative ones).
template <int Q>
__device__ __forceinline__ int fx_line_max(const long long (&x)[Q]) {
    int hi = (int)(x[0] >> 32), lo = hi;
#pragma unroll
    for (int l = 1; l < Q; l += 2) {
        const int a = (int)(x[l] >> 32), b = (l + 1 < Q) ? (int)(x[l + 1 < Q ? l + 1 : l] >> 32) : a;
        hi = __vimax3_s32(hi, a, b);
        lo = __vimin3_s32(lo, a, b);
    }
    return max(hi, ~lo);
}

// *slot = max(*slot, v) over the `lines` threads of an element (consecutive
// threads): once per warp where the element is made of whole warps.
template <int lines>
__device__ __forceinline__ void fx_element_max(unsigned *slot, unsigned v) {
    if constexpr (lines % 32 == 0) {
        v = __reduce_max_sync(0xffffffffu, v);
        if (threadIdx.x % 32 == 0) atomicMax(slot, v);
    } else {
        atomicMax(slot, v);
    }
}

// The FP64 counterpart for the elements that the fixed-point path leaves out:
// y = A x along a line, A folded at c_fold[OFF].  The operator entries come
// from global memory (the constant bank holds the fixed-point tables); the
// FP64 pipe takes 16 clocks per warp instruction and SM, behind which a load
// for each hides.  Every rounding is written out (no contraction left to the
// compiler): an element has the same bits in each kernel that computes it.
template <int P, int Q, int SIG, int OFF, class F>
__device__ __forceinline__ void fx_line64(const double (&x)[Q], F &&put) {
    constexpr int hp = P / 2, hq = Q / 2;
    constexpr int oS = OFF, oT = OFF + hp * hq, oC = OFF + 2 * hp * hq;
    constexpr int oR = oC + ((Q % 2) ? hp : 0);
    double e[hq], o[hq];
#pragma unroll
    for (int i = 0; i < hq; i++) {
        e[i] = x[i] + x[Q - 1 - i];
        o[i] = x[i] - x[Q - 1 - i];
    }
#pragma unroll
    for (int a = 0; a < hp; a++) {
        double E = __dmul_rn(__ldg(c_fold + oS + a * hq), e[0]), O = __dmul_rn(__ldg(c_fold + oT + a * hq), o[0]);
#pragma unroll
        for (int i = 1; i < hq; i++) {
            E = fma(__ldg(c_fold + oS + a * hq + i), e[i], E);
            O = fma(__ldg(c_fold + oT + a * hq + i), o[i], O);
        }
        if (Q % 2) E = fma(__ldg(c_fold + oC + a), x[hq], E);
        put(a, E + O);
        put(P - 1 - a, (SIG > 0) ? (E - O) : (O - E));
    }
    if (P % 2) {
        double M = __dmul_rn(__ldg(c_fold + oR), (SIG > 0) ? e[0] : o[0]);
#pragma unroll
        for (int i = 1; i < hq; i++) M = fma(__ldg(c_fold + oR + i), (SIG > 0) ? e[i] : o[i], M);
        if ((Q % 2) && SIG > 0) M = fma(__ldg(c_fold + oR + hq), x[hq], M);
        put(hp, M);
    }
}

// (a x + b y + c z) in FP64, rounded as written.
__device__ __forceinline__ double fx_dot64(double a, double x, double b, double y, double c, double z) {
    return fma(c, z, fma(b, y, __dmul_rn(a, x)));
}

#define FEM_DEFINE_FX_UPLOAD(NAME)                                                                        \
    cudaError_t NAME(const double *table) {                                                               \
        const FxTables &t = fx_tables();                                                                  \
        cudaError_t e = cudaMemcpyToSymbol(c_fx, t.c, sizeof(t.c), 0, cudaMemcpyHostToDevice);            \
        if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_fxd, t.d, sizeof(t.d), 0, cudaMemcpyHostToDevice); \
        if (e != cudaSuccess) return e;                                                                   \
        return cudaMemcpyToSymbol(c_fold, table, sizeof(double) * kFoldTotal, 0, cudaMemcpyHostToDevice); \
    }

}  // namespace fem
