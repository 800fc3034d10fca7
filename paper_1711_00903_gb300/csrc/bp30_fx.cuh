// BP1.0, BP3.0 and both in one pass in FP64 with their arithmetic on the
// integer multiply-add pipe (fx.cuh), shared by the stand-alone kernels
// (bp1_fx.cu, bp30_fx.cu) and the batched persistent kernel (batch.cu).
//
// The scales follow the element's data as in bp35_fx.cuh:
//   1. q, scaled by the element's largest |q| to 59 or 60 bits, through the
//      three interpolations (each output is a mix of the whole element, so
//      one scale serves it), scaled up once more before the third;
//   2. BP1.0: times wJ (62 bits, without its weights' powers of two), through
//      the three projections, which carry the weights: the second takes its
//      input scaled up by the element's largest value, the third by the
//      line's (three in a row at the worst case's scale would lose 6 to 9
//      bits);
//   3. BP3.0: derivatives, scaled up by their largest value; chain rule with
//      the factors scaled to 62 bits (on flat elements direction by direction,
//      FxScales); transposes, each line scaled up by its
//      largest value; their sum with lambda wJ q, aligned, scaled up by its
//      largest value; the three projections.
// BP1.0 computed beside BP3.0 takes the same steps on the same numbers as
// alone, and BP3.0 the same with and without it: equal bits.
//
// An element goes through FP64 instead (bp1_left64, bp30_left64) when its values
// are not finite or extreme, when one of its eight octants holds no value near
// its largest (the FP64 result there would keep digits that the element's scale
// cuts off), when a point's factors are far below the element's largest, when the
// factors are not positive definite or, at N = 1, when the lines hold far less
// than their directions' scale; element by element, so a result does not depend
// on the block's other elements.
// What the field or a factor's sign tells, it tells before the contractions; a
// mesh of such elements takes 0.9 to 1.06 of the FP64 kernels' time.
//
// What bounds it: integer multiply-adds and, between barriers, latency; see
// bp30_fx.cu and bp1_fx.cu for the measured rates.  The error against quadruple
// precision on jittered elements is 0.05 to 0.47 of the FP64 lines' (BP3.0),
// 0.13 to 0.59 (BP1.0).
#pragma once

#include "bp30_body.cuh"  // Bp30Layout
#include "fx.cuh"
#include "fx_point.cuh"

namespace fem {
namespace {

// How far (in bits) below the element's largest value an octant's largest
// may lie.  At N = 1, where an octant is one node (of a field that vanishes
// on a face, a zero), every node's result holds at least an eighth of every
// other's: any range will do.
__host__ __device__ constexpr int fx30_octant_range(int N) { return N == 1 ? 2047 : kFxRange; }

// Slots of an element's statistics: the eight octants of q, the largest wJ,
// Grr, Gss, Gtt, derivatives along r, s, t (FxScales) and sum at the Gauss
// points, whether the element is left to FP64 (BP1.0, BP3.0), the largest value
// after the projection along t (BP1.0, BP3.0) and after the interpolation along
// s, the largest scale of a transposed line (as 63 - its scale-up) and of the
// direction of one that is not zero (N = 1), the directions' scales (fx_below).
enum {
    kFxW = 8, kFxG = 9, kFxU = 12, kFxX = 15, kFxLeft1 = 16, kFxLeft30 = 17, kFxT1 = 18, kFxT30 = 19, kFxI = 20, kFxH = 21,
    kFxE = 22, kFxB = 23, kFx30Stats = 24
};

// A line of Q values at from(l), contracted, its outputs to put(l, y).
template <int P, int Q, int SIG, int OFF, class L, class F>
__device__ __forceinline__ void fx_line(L &&from, F &&put) {
    long long x[Q];
#pragma unroll
    for (int l = 0; l < Q; l++) x[l] = from(l);
    fx_apply<P, Q, SIG, OFF>(x, put);
}

// g x / 2^62 of a factor below 2^62 (halves) and |x| < 2^60.
__device__ __forceinline__ long long fx_mul(int gh, int gl, long long x) {
    const int xh = fx_hi(x), xl = fx_lo(x);
    return (mul_wide(gh, xh) << 2) + (mad_wide(gl, xh, mad_wide(gh, xl, 1ll << 29)) >> 30);
}

// Scale-up of the values before the interpolation along t.
template <int N>
__device__ __forceinline__ int fx30_up(const unsigned *st) {
    return max(0, fx_qbits30(N) - 32 - fx_top((int)st[kFxI]));
}

// The high word's largest magnitude over the values seen.
struct FxMost {
    int hi = 0, lo = 0;
    __device__ __forceinline__ void see(long long x) {
        hi = max(hi, (int)(x >> 32));
        lo = min(lo, (int)(x >> 32));
    }
    __device__ __forceinline__ int value() const { return max(hi, ~lo); }
};

// The projections of EPB elements along s (box X of t-projected values, whose
// largest is at `slot` of the statistics, to box Y) and along r (box Y to the
// output, exponent(e) that of the s-projected values without their scale-up),
// for elements not left to FP64.
template <int N, int EPB_, class B1, class B2>
__device__ __forceinline__ void fx30_project_s(int nel, const long long *X, long long *Y, int per, const unsigned *stats,
                                               int slot) {
    constexpr int n = N + 1, m = N + 2;
    for_tasks<m * n, EPB_>(nel, [&](int e, int t) {
        const long long *Xe = X + e * per;
        long long *Ye = Y + e * per;
        const int i = t % m, k = t / m, up = max(0, kFxBits30 - 32 - fx_top((int)stats[e * kFx30Stats + slot]));
        fx_line<n, m, 1, fold_offset(N, kFoldIT)>([&](int l) { return Xe[B2::at(i, l, k)] << up; },
                                                  [&](int l, long long y) { Ye[B1::at(i, l, k)] = y; });
    });
}
template <int N, int EPB_, class B1, class F, class O>
__device__ __forceinline__ void fx30_project_r(int nel, const long long *Y, int per, const unsigned *stats, int slot,
                                               int left, F &&exponent, O &&out) {
    constexpr int n = N + 1, m = N + 2;
    for_tasks<n * n, EPB_>(nel, [&](int e, int t) {
        const unsigned *se = stats + e * kFx30Stats;
        if (se[left] != 0) return;
        const long long *Ye = Y + e * per;
        const int j = t % n, k = t / n;
        long long x[m];
#pragma unroll
        for (int l = 0; l < m; l++) x[l] = Ye[B1::at(l, j, k)];
        const int h = max(0, kFxBits30 - 32 - fx_top(fx_line_max(x)));
#pragma unroll
        for (int l = 0; l < m; l++) x[l] <<= h;
        const int k2 = exponent(e) - max(0, kFxBits30 - 32 - fx_top((int)se[slot])) - h + c_fxd[N].wn[j] + c_fxd[N].wn[k];
        fx_apply<n, m, 1, fold_offset(N, kFoldIT)>(
            x, [&](int l, long long y) { out(e, t, l, fx_to_double(y, k2 + c_fxd[N].wn[l])); });
    });
}

// Loads the field of column (i, j) = r of an element (r < n^2; PCG: p <- z +
// beta p, stored) and folds its largest values into the octants' slots; a
// middle node belongs to both halves.
template <int N, bool PCG>
__device__ __forceinline__ void fx30_load(double (&qv)[N + 1], int64_t g0, int r, const double *__restrict__ q,
                                          const double *__restrict__ z, double *p, const double *__restrict__ beta,
                                          unsigned *st) {
    constexpr int n = N + 1, nn = n * n;
    if (PCG) {
        const double bt = *beta;
#pragma unroll
        for (int k = 0; k < n; k++) {
            const int64_t g = g0 + k * nn;
            qv[k] = (bt == 0.0) ? z[g] : fma(bt, p[g], z[g]);
            p[g] = qv[k];
        }
    } else {
#pragma unroll
        for (int k = 0; k < n; k++) qv[k] = __ldg(q + g0 + k * nn);
    }
    unsigned lo = 0, hi = 0;
#pragma unroll
    for (int k = 0; k < n; k++) {
        const unsigned a = (unsigned)fx_abs_hi(qv[k]);
        if (k <= N / 2) lo = max(lo, a);
        if (k >= n / 2) hi = max(hi, a);
    }
    const int i = r % n, j = r / n;
#pragma unroll
    for (int o = 0; o < 4; o++) {
        const bool in_i = (o & 1) ? i >= n / 2 : i <= N / 2, in_j = (o & 2) ? j >= n / 2 : j <= N / 2;
        if (in_i && in_j) {
            atomicMax(st + o, lo);
            atomicMax(st + 4 + o, hi);
        }
    }
}

// High word (so: sign) of a factor that has to be positive, read ahead with the
// field by an element's first thread: an element of a left-handed mesh has them
// all negative, and is left to FP64 before its contractions.
__device__ __forceinline__ int fx30_sign(const double *g) { return __ldg(reinterpret_cast<const int *>(g) + 1); }

// The element's scale from its octants: |q| < 2^kq; left: the element is not
// held to one scale.
template <int N>
__device__ __forceinline__ int fx30_scale(const unsigned *st, bool *left) {
    unsigned most = 0, least = 0x7fffffffu;
#pragma unroll
    for (int o = 0; o < 8; o++) {
        most = max(most, st[o]);
        least = min(least, st[o]);
    }
    const int e = (int)(most >> 20);
    *left = most != 0 && (e < 64 || e == 0x7ff || (int)(least >> 20) < e - fx30_octant_range(N));
    return most ? e - 1022 : 0;
}

// Largest exponents (high words without the weights) of `planes` factor
// planes at column r of the Gauss points (weights of the column wab).
template <int N, int planes>
__device__ __forceinline__ void fx30_scan(const double *Ge, const int (&plane)[planes], int wab, unsigned *slots) {
    constexpr int m = N + 2, mm = m * m, MP = m * mm;
    const int *Gi = reinterpret_cast<const int *>(Ge) + 1;  // high words
    int most[planes];
#pragma unroll
    for (int h = 0; h < planes; h++) most[h] = 0;
#pragma unroll 4
    for (int c = 0; c < m; c++) {
        const int w = c_fxd[N].wm[c] << 20;
#pragma unroll
        for (int h = 0; h < planes; h++) most[h] = max(most[h], __ldg(Gi + 2 * (plane[h] * MP + c * mm)) - w);
    }
#pragma unroll
    for (int h = 0; h < planes; h++) fx_element_max<mm>(slots + h, (unsigned)(most[h] - (wab << 20)));
}

// BP1.0's step at a Gauss point: wJ qg, with wJ scaled by 2^(62 - kw).
// bw: kw + 1022 plus the point's weight exponents.  A wJ that is not positive
// or far below the element's largest raises far, a larger or non-finite one
// lowers least.
__device__ __forceinline__ long long fx30_mass(double wj, int bw, long long qg, int &far, int &least) {
    const int s = bw - (__double2hiint(wj) >> 20);
    far = max(far, s);
    least = min(least, s);
    int gh, gl;
    fx_diagonal(wj, s, gh, gl);
    return fx_mul(gh, gl, qg);
}

// Exponent of BP1.0's projected values (without the scale-ups) from an
// element's statistics.
template <int N>
__device__ __forceinline__ int fx1_exponent(const unsigned *st) {
    bool left;
    return fx30_scale<N>(st, &left) - fx_qbits30(N) - fx30_up<N>(st) + 3 * (c_fxd[N].tau[kFoldI] + c_fxd[N].tau[kFoldIT]) +
           (int)(st[kFxW] >> 20) - 1022;
}

// A line of doubles at from(l), contracted in FP64, its outputs to put(l, y).
template <int P, int Q, int SIG, int OFF, class L, class F>
__device__ __forceinline__ void fx_from64(L &&from, F &&put) {
    double x[Q];
#pragma unroll
    for (int l = 0; l < Q; l++) x[l] = from(l);
    fx_line64<P, Q, SIG, OFF>(x, put);
}

// In FP64, of the block's elements for which on(e) holds: the interpolation
// along r (box X to Y) and s (Y to X), between barriers.
template <int N, int EPB_, class B0, class B1, class B2, class F>
__device__ __forceinline__ void fx30_interpolate64(int nel, double *X, double *Y, int per, F &&on) {
    constexpr int n = N + 1, m = N + 2, oI = fold_offset(N, kFoldI);
    for_tasks<n * n, EPB_>(nel, [&](int e, int t) {
        if (!on(e)) return;
        const double *x = X + e * per;
        double *y = Y + e * per;
        const int j = t % n, k = t / n;
        fx_from64<m, n, 1, oI>([&](int l) { return x[B0::at(l, j, k)]; }, [&](int l, double w) { y[B1::at(l, j, k)] = w; });
    });
    __syncthreads();
    for_tasks<m * n, EPB_>(nel, [&](int e, int t) {
        if (!on(e)) return;
        const double *y = Y + e * per;
        double *x = X + e * per;
        const int i = t % m, k = t / m;
        fx_from64<m, n, 1, oI>([&](int l) { return y[B1::at(i, l, k)]; }, [&](int l, double w) { x[B2::at(i, l, k)] = w; });
    });
    __syncthreads();
}

// The projection along s (box X to Y) and r (Y to out(e, t, l, value)).
template <int N, int EPB_, class B1, class B2, class F, class O>
__device__ __forceinline__ void fx30_project64(int nel, const double *X, double *Y, int per, F &&on, O &&out) {
    constexpr int n = N + 1, m = N + 2, oIT = fold_offset(N, kFoldIT);
    for_tasks<m * n, EPB_>(nel, [&](int e, int t) {
        if (!on(e)) return;
        const double *x = X + e * per;
        double *y = Y + e * per;
        const int i = t % m, k = t / m;
        fx_from64<n, m, 1, oIT>([&](int l) { return x[B2::at(i, l, k)]; }, [&](int l, double w) { y[B1::at(i, l, k)] = w; });
    });
    __syncthreads();
    for_tasks<n * n, EPB_>(nel, [&](int e, int t) {
        if (!on(e)) return;
        const double *y = Y + e * per;
        const int j = t % n, k = t / n;
        fx_from64<n, m, 1, oIT>([&](int l) { return y[B1::at(l, j, k)]; }, [&](int l, double w) { out(e, t, l, w); });
    });
}

// ---------------------------------------------------------------- BP1.0

// Shared memory of EPB elements: a box for q, the twice interpolated and the
// once projected field, one for the once interpolated and the twice
// projected, the statistics and two flags of the block: an element is on the
// fixed-point path; one is left to FP64.
template <int N, int EPB_>
struct Fx1Layout {
    static constexpr int n = N + 1, m = N + 2, nn = n * n, mm = m * m, NP = nn * n, MP = mm * m, EPB = EPB_;
    using B0 = Box<n, n, n>;
    using B1 = Box<m, n, n>;
    using B2 = Box<m, m, n>;
    static constexpr int SA = B0::size > B2::size ? B0::size : B2::size, per = SA + B1::size;
    static constexpr int threads = ((mm * EPB + 31) / 32) * 32;
    static constexpr int off_stats = EPB * per * 8;
    static constexpr int off_b = off_stats + EPB * kFx30Stats * 4;  // the block's flags
    static constexpr int smem = off_b + 8;
};

// Algorithm 3 in FP64 on the elements left to it, all at once, in the boxes of
// the fixed-point path.  A function of its own: its registers are not that path's.
template <int N, int EPB_>
__device__ __noinline__ void bp1_left64(unsigned char *smem_raw, int64_t e0, int nel, const double *wJ, const double *q,
                                        double *Mq) {
    using C = Fx1Layout<N, EPB_>;
    using B0 = typename C::B0;
    using B2 = typename C::B2;
    constexpr int n = C::n, m = C::m, nn = C::nn, mm = C::mm, NP = C::NP, MP = C::MP;
    const unsigned *stats = reinterpret_cast<const unsigned *>(smem_raw + C::off_stats);
    double *X = reinterpret_cast<double *>(smem_raw), *Y = X + C::SA;
    auto on = [&](int e) { return stats[e * kFx30Stats + kFxLeft1] != 0; };
    const int el = threadIdx.x / mm, r = threadIdx.x - el * mm;
    const bool act = el < nel && on(el);
    __syncthreads();  // the shared memory is free
    if (act && r < nn) {
#pragma unroll
        for (int k = 0; k < n; k++) X[el * C::per + B0::at(r % n, r / n, k)] = __ldg(q + (e0 + el) * NP + r + k * nn);
    }
    __syncthreads();
    fx30_interpolate64<N, EPB_, B0, typename C::B1, B2>(nel, X, Y, C::per, on);
    if (act) {
        double *x = X + el * C::per, w[m];
        const double *we = wJ + (e0 + el) * MP + r;
        const int a = r % m, b = r / m;
        fx_from64<m, n, 1, fold_offset(N, kFoldI)>([&](int l) { return x[B2::at(a, b, l)]; },
                                                   [&](int c, double g) { w[c] = __dmul_rn(g, __ldg(we + c * mm)); });
        fx_line64<n, m, 1, fold_offset(N, kFoldIT)>(w, [&](int l, double y) { x[B2::at(a, b, l)] = y; });
    }
    __syncthreads();
    fx30_project64<N, EPB_, typename C::B1, B2>(nel, X, Y, C::per, on, [&](int e, int t, int l, double w) {
        Mq[(e0 + e) * NP + t * n + l] = w;
    });
}

// BP1.0 of elements [e0, e0 + nel) by the whole block (blockDim.x >=
// Layout::threads); wJ: m^3 values per element.
template <int N, int EPB_>
__device__ __forceinline__ void bp1_fx_block(unsigned char *smem_raw, int64_t e0, int nel, const double *__restrict__ wJ,
                                             const double *__restrict__ q, double *__restrict__ Mq) {
    using C = Fx1Layout<N, EPB_>;
    using B0 = typename C::B0;
    using B1 = typename C::B1;
    using B2 = typename C::B2;
    constexpr int n = C::n, m = C::m, nn = C::nn, mm = C::mm, NP = C::NP, MP = C::MP, K = kFx30Stats, QB = fx_qbits30(N);
    constexpr int oI = fold_offset(N, kFoldI), oIT = fold_offset(N, kFoldIT);
    const int el = threadIdx.x / mm, r = threadIdx.x - el * mm;
    const bool act = el < nel;
    const int a = r % m, b = r / m;
    long long *boxes = reinterpret_cast<long long *>(smem_raw);
    unsigned *stats = reinterpret_cast<unsigned *>(smem_raw + C::off_stats), *st = stats + el * K;
    if (threadIdx.x == 0) prefetch_l2(wJ + e0 * MP, (long long)nel * MP * 8);
    volatile unsigned *flag = reinterpret_cast<volatile unsigned *>(smem_raw + C::off_b);
    for (int t = threadIdx.x; t < EPB_ * K + 2; t += blockDim.x) stats[t] = 0;  // (the flags lie behind them)
    __syncthreads();

    double qv[n];
    const bool col = act && r < nn;
    const int sign = act && r == 0 ? fx30_sign(wJ + (e0 + el) * MP) : 0;
    if (col) fx30_load<N, false>(qv, (e0 + el) * NP + r, r, q, nullptr, nullptr, nullptr, st);
    __syncthreads();
    int kq = 0;
    if (act) {
        bool left;
        kq = fx30_scale<N>(st, &left);
        left = left || sign < 0;
        if (col) {
#pragma unroll
            for (int k = 0; k < n; k++) {
                const int e = (__double2hiint(qv[k]) >> 20) & 0x7ff;
                left = left || (kq == 0 && e == 0 && (fx_abs_hi(qv[k]) | __double2loint(qv[k])) != 0);
                boxes[el * C::per + B0::at(r % n, r / n, k)] = fx_from_double<QB>(qv[k], kq + 1022 - e);
            }
        }
        if (left) st[kFxLeft1] = 1;
        if (left) flag[1] = 1;
        if (!left && r == 0) flag[0] = 1;
    }
    __syncthreads();
    if (flag[0] != 0) {
        // interpolation along r and s
        for_tasks<nn, EPB_>(nel, [&](int e, int t) {
            const long long *X = boxes + e * C::per;
            long long *Y = boxes + e * C::per + C::SA;
            const int j = t % n, k = t / n;
            fx_line<m, n, 1, oI>([&](int l) { return X[B0::at(l, j, k)]; }, [&](int l, long long y) { Y[B1::at(l, j, k)] = y; });
        });
        const int wab = act ? c_fxd[N].wm[a] + c_fxd[N].wm[b] : 0;
        if (act) fx30_scan<N, 1>(wJ + (e0 + el) * MP + r, {0}, wab, st + kFxW);
        __syncthreads();
        for_tasks<m * n, EPB_>(nel, [&](int e, int t) {
            const long long *Y = boxes + e * C::per + C::SA;
            long long *X = boxes + e * C::per;
            const int i = t % m, k = t / m;
            FxMost most;
            fx_line<m, n, 1, oI>([&](int l) { return Y[B1::at(i, l, k)]; },
                                 [&](int l, long long y) {
                                     X[B2::at(i, l, k)] = y;
                                     most.see(y);
                                 });
            atomicMax(stats + e * K + kFxI, (unsigned)most.value());
        });
        __syncthreads();

        // column (a, b): interpolation, wJ and projection along t
        if (act) {
            long long *X = boxes + el * C::per, w[m];
            const int kw = (int)(st[kFxW] >> 20) - 1022, bw = kw + 1022 + wab;
            int far = 0, least = 0;
            const double *we = wJ + (e0 + el) * MP + r;
            const int up = fx30_up<N>(st);
            fx_line<m, n, 1, oI>([&](int l) { return X[B2::at(a, b, l)] << up; },
                                 [&](int c, long long g) {
                                     w[c] = fx30_mass(__ldg(we + c * mm), bw + c_fxd[N].wm[c], g, far, least);
                                 });
            FxMost most;
            fx_apply<n, m, 1, oIT>(w, [&](int l, long long y) {
                X[B2::at(a, b, l)] = y;
                most.see(y);
            });
            fx_element_max<mm>(st + kFxT1, (unsigned)most.value());
            if (least < 0 || far > kFxRange || kw > 800 || kw < -800 || kq + kw > 800 || kq + kw < -800)
                st[kFxLeft1] = flag[1] = 1;
        }
        __syncthreads();

        // projection along s and r
        fx30_project_s<N, EPB_, B1, B2>(nel, boxes, boxes + C::SA, C::per, stats, kFxT1);
        __syncthreads();
        fx30_project_r<N, EPB_, B1>(
            nel, boxes + C::SA, C::per, stats, kFxT1, kFxLeft1, [&](int e) { return fx1_exponent<N>(stats + e * K); },
            [&](int e, int t, int l, double w) { Mq[(e0 + e) * NP + t * n + l] = w; });
    }
    if (flag[1] != 0) bp1_left64<N, EPB_>(smem_raw, e0, nel, wJ, q, Mq);
}

// ---------------------------------------------------------------- BP3.0

// Shared memory of EPB elements: four m^3 boxes, a word per line, the
// statistics, the block's flags (as in Fx1Layout).
template <int N, int EPB_>
struct Fx30Layout {
    static constexpr int n = N + 1, m = N + 2, nn = n * n, mm = m * m, NP = nn * n, MP = mm * m, EPB = EPB_;
    using B0 = Box<n, n, n>;
    using B1 = Box<m, n, n>;
    using B2 = Box<m, m, n>;
    using B3 = Box<m, m, m>;
    static constexpr int S = B3::size, per = 4 * S;
    static constexpr int threads = ((mm * EPB + 31) / 32) * 32;
    static constexpr int off_e = EPB * per * 8;
    static constexpr int off_s = off_e + EPB * 3 * mm * 4;
    static constexpr int off_b = off_s + EPB * kFx30Stats * 4;  // the block's flags
    static constexpr int smem_ = off_b + 8;
    static constexpr int smem = smem_ > threads * 8 ? smem_ : threads * 8;
};

// Algorithm 5 (MASS: and Algorithm 3) in FP64 on the elements left to it, all at
// once, in the boxes of the fixed-point path.  Returns the thread's share of q . Aq.
template <int N, int EPB_, bool MASS>
__device__ __noinline__ double bp30_left64(unsigned char *smem_raw, int64_t e0, int nel, const double *G, double lambda,
                                           const double *q, double *Aq, double *Mq) {
    using C = Fx30Layout<N, EPB_>;
    using B0 = typename C::B0;
    using B1 = typename C::B1;
    using B2 = typename C::B2;
    using B3 = typename C::B3;
    constexpr int n = C::n, m = C::m, nn = C::nn, mm = C::mm, NP = C::NP, MP = C::MP, S = C::S, per = C::per;
    constexpr int oI = fold_offset(N, kFoldI), oIT = fold_offset(N, kFoldIT);
    constexpr int oDt = fold_offset(N, kFoldDt), oDtT = fold_offset(N, kFoldDtT);
    const unsigned *stats = reinterpret_cast<const unsigned *>(smem_raw + C::off_s);
    double *boxes = reinterpret_cast<double *>(smem_raw);
    auto on30 = [&](int e) { return stats[e * kFx30Stats + kFxLeft30] != 0; };
    auto on1 = [&](int e) { return MASS && stats[e * kFx30Stats + kFxLeft1] != 0; };
    auto on = [&](int e) { return on30(e) || on1(e); };
    const int el = threadIdx.x / mm, r = threadIdx.x - el * mm, u = r % m, v = r / m;
    const bool act = el < nel && on(el), act30 = el < nel && on30(el);
    double *A = boxes + el * per, *B = A + S, *Cx = B + S, *D = Cx + S;
    const double *Ge = G + (e0 + el) * 7 * MP + r;
    __syncthreads();  // the shared memory is free
    if (act && r < nn) {
#pragma unroll
        for (int k = 0; k < n; k++) B[B0::at(r % n, r / n, k)] = q[(e0 + el) * NP + r + k * nn];
    }
    __syncthreads();
    // interpolation along r (B -> C), s (C -> B) and t (B -> A)
    fx30_interpolate64<N, EPB_, B0, B1, B2>(nel, boxes + S, boxes + 2 * S, per, on);
    if (act)
        fx_from64<m, n, 1, oI>([&](int l) { return B[B2::at(u, v, l)]; }, [&](int l, double y) { A[B3::at(u, v, l)] = y; });
    __syncthreads();
    if constexpr (MASS) {  // wJ and projection (A -> B -> C -> Mq)
        if (act && on1(el))
            fx_from64<n, m, 1, oIT>([&](int c) { return __dmul_rn(A[B3::at(u, v, c)], __ldg(Ge + 6 * MP + c * mm)); },
                                    [&](int l, double y) { B[B2::at(u, v, l)] = y; });
        __syncthreads();
        fx30_project64<N, EPB_, B1, B2>(nel, boxes + S, boxes + 2 * S, per, on1, [&](int e, int t, int l, double w) {
            Mq[(e0 + e) * NP + t * n + l] = w;
        });
        __syncthreads();
    }
    // derivatives along r (A -> B), s (A -> C) and t (A -> D); the directions take
    // turns in one loop (side by side they spilled)
    auto line = [&](auto off, int d, const double *from, double *to) {
        const int step = d == 0 ? 1 : d == 1 ? B3::sj : B3::sk,
                  at = d == 0 ? B3::at(0, u, v) : d == 1 ? B3::at(u, 0, v) : B3::at(u, v, 0);
        fx_from64<m, m, -1, off.value>([&](int l) { return from[at + l * step]; },
                                       [&](int l, double y) { to[at + l * step] = y; });
    };
    using Dt = std::integral_constant<int, oDt>;
    using DtT = std::integral_constant<int, oDtT>;
    if (act30) {
#pragma unroll 1
        for (int d = 0; d < 3; d++) line(Dt(), d, A, B + d * S);
    }
    __syncthreads();
    if (act30) {
#pragma unroll 2
        for (int c = 0; c < m; c++) {
            const int s = B3::at(u, v, c);
            const double *g = Ge + c * mm, qr = B[s], qs = Cx[s], qt = D[s], g1 = __ldg(g + MP), g2 = __ldg(g + 2 * MP),
                         g4 = __ldg(g + 4 * MP);
            B[s] = fx_dot64(__ldg(g), qr, g1, qs, g2, qt);
            Cx[s] = fx_dot64(g1, qr, __ldg(g + 3 * MP), qs, g4, qt);
            D[s] = fx_dot64(g2, qr, g4, qs, __ldg(g + 5 * MP), qt);
        }
    }
    __syncthreads();
    if (act30) {
#pragma unroll 1
        for (int d = 0; d < 3; d++) line(DtT(), d, B + d * S, B + d * S);
    }
    __syncthreads();
    // column: the three directions, lambda wJ q and projection along t (D in place), s (D -> C) and r (C -> Aq)
    if (act30)
        fx_from64<n, m, 1, oIT>(
            [&](int c) {
                const int s = B3::at(u, v, c);
                double w = D[s];
                if (lambda != 0.0) w = fma(__dmul_rn(lambda, __ldg(Ge + 6 * MP + c * mm)), A[s], w);
                return w + (B[s] + Cx[s]);
            },
            [&](int l, double y) { D[B2::at(u, v, l)] = y; });
    __syncthreads();
    double dot = 0.0;
    fx30_project64<N, EPB_, B1, B2>(nel, boxes + 3 * S, boxes + 2 * S, per, on30, [&](int e, int t, int l, double w) {
        const int64_t g = (e0 + e) * NP + t * n + l;
        Aq[g] = w;
        dot = fma(q[g], w, dot);
    });
    return dot;
}

// BP3.0 of elements [e0, e0 + nel) by the whole block (blockDim.x >=
// Layout::threads); MASS: BP1.0 too, to Mq, with wJ the seventh factor.  PCG
// as bp35_block.
template <int N, int EPB_, bool PCG, bool MASS>
__device__ __forceinline__ void bp30_fx_block(unsigned char *smem_raw, int64_t e0, int nel, const double *__restrict__ G,
                                              double lambda, const double *__restrict__ q, double *__restrict__ Aq,
                                              double *__restrict__ Mq, const double *__restrict__ z, double *p,
                                              const double *__restrict__ beta, double *__restrict__ part_out) {
    using C = Fx30Layout<N, EPB_>;
    using B0 = typename C::B0;
    using B1 = typename C::B1;
    using B2 = typename C::B2;
    using B3 = typename C::B3;
    constexpr int n = C::n, m = C::m, nn = C::nn, mm = C::mm, NP = C::NP, MP = C::MP, S = C::S, K = kFx30Stats, QB = kFxBits30, qb = fx_qbits30(N);
    constexpr int oI = fold_offset(N, kFoldI), oIT = fold_offset(N, kFoldIT);
    constexpr int oDt = fold_offset(N, kFoldDt), oDtT = fold_offset(N, kFoldDtT);
    constexpr bool EXACT = N == 1;  // FP64 may interpolate and differentiate without an error
    const int el = threadIdx.x / mm, r = threadIdx.x - el * mm;
    const bool act = el < nel;
    const int u = r % m, v = r / m;
    long long *boxes = reinterpret_cast<long long *>(smem_raw);
    long long *A = boxes + el * C::per, *B = A + S, *Cx = B + S, *D = Cx + S;
    int *ln = reinterpret_cast<int *>(smem_raw + C::off_e) + el * 3 * mm;
    unsigned *stats = reinterpret_cast<unsigned *>(smem_raw + C::off_s), *st = stats + el * K;
    if (threadIdx.x == 0) prefetch_l2(G + e0 * 7 * MP, (long long)nel * 7 * MP * 8);
    volatile unsigned *flag = reinterpret_cast<volatile unsigned *>(smem_raw + C::off_b);
    for (int t = threadIdx.x; t < EPB_ * K + 2; t += blockDim.x) stats[t] = 0;  // (the flags lie behind them)
    __syncthreads();

    double qv[n];
    const bool col = act && r < nn;
    const double *Ge = G + (e0 + el) * 7 * MP + r;
    const int sign = act && r == 0 ? fx30_sign(Ge) : 0, sign1 = MASS && act && r == 0 ? fx30_sign(Ge + 6 * MP) : 0;
    if (col) fx30_load<N, PCG>(qv, (e0 + el) * NP + r, r, q, z, p, beta, st);
    __syncthreads();
    int kq = 0;
    if (act) {
        bool left;
        kq = fx30_scale<N>(st, &left);
        if (col) {
#pragma unroll
            for (int k = 0; k < n; k++) {
                const int e = (__double2hiint(qv[k]) >> 20) & 0x7ff;
                left = left || (kq == 0 && e == 0 && (fx_abs_hi(qv[k]) | __double2loint(qv[k])) != 0);
                B[B0::at(r % n, r / n, k)] = fx_from_double<qb>(qv[k], kq + 1022 - e);
            }
        }
        if (left || sign1 < 0) st[kFxLeft1] = 1;
        if (left || sign < 0) st[kFxLeft30] = 1;
        if (left || sign < 0 || sign1 < 0) flag[1] = 1;
        if (r == 0 && !left && (sign >= 0 || (MASS && sign1 >= 0))) flag[0] = 1;
    }
    __syncthreads();
    double dot = 0.0;  // p . Ap of the thread's lines
    if (flag[0] != 0) {
        // interpolation along r (B -> C), s (C -> B) and t (B -> A)
        for_tasks<nn, EPB_>(nel, [&](int e, int t) {
            const long long *X = boxes + e * C::per + S;
            long long *Y = boxes + e * C::per + 2 * S;
            const int j = t % n, k = t / n;
            fx_line<m, n, 1, oI>([&](int l) { return X[B0::at(l, j, k)]; }, [&](int l, long long y) { Y[B1::at(l, j, k)] = y; });
        });
        __syncthreads();
        for_tasks<m * n, EPB_>(nel, [&](int e, int t) {
            const long long *Y = boxes + e * C::per + 2 * S;
            long long *X = boxes + e * C::per + S;
            const int i = t % m, k = t / m;
            FxMost most;
            fx_line<m, n, 1, oI>([&](int l) { return Y[B1::at(i, l, k)]; },
                                 [&](int l, long long y) {
                                     X[B2::at(i, l, k)] = y;
                                     most.see(y);
                                 });
            atomicMax(stats + e * K + kFxI, (unsigned)most.value());
        });
        __syncthreads();
        const int wuv = act ? c_fxd[N].wm[u] + c_fxd[N].wm[v] : 0;
        int t3 = 3 * c_fxd[N].tau[kFoldI];  // exponent of the interpolated field over q's
        if (act) {
            t3 -= fx30_up<N>(st);
            const int up = fx30_up<N>(st);
            fx_line<m, n, 1, oI>([&](int l) { return B[B2::at(u, v, l)] << up; },
                                 [&](int l, long long y) { A[B3::at(u, v, l)] = y; });
            fx30_scan<N, 4>(Ge, {6, 0, 3, 5}, wuv, st + kFxW);
        }
        __syncthreads();
        const int kw = act ? (int)(st[kFxW] >> 20) - 1022 : 0;

        // BP1.0: wJ and projection along t (A -> B), s (B -> C) and r (C -> Mq)
        if constexpr (MASS) {
            if (act) {
                long long w[m];
                const int bw = kw + 1022 + wuv;
                int far = 0, least = 0;
#pragma unroll
                for (int c = 0; c < m; c++)
                    w[c] = fx30_mass(__ldg(Ge + 6 * MP + c * mm), bw + c_fxd[N].wm[c], A[B3::at(u, v, c)], far, least);
                FxMost most;
                fx_apply<n, m, 1, oIT>(w, [&](int l, long long y) {
                    B[B2::at(u, v, l)] = y;
                    most.see(y);
                });
                fx_element_max<mm>(st + kFxT1, (unsigned)most.value());
                if (least < 0 || far > kFxRange || kw > 800 || kw < -800 || kq + kw > 800 || kq + kw < -800)
                    st[kFxLeft1] = flag[1] = 1;
            }
            __syncthreads();
            fx30_project_s<N, EPB_, B1, B2>(nel, boxes + S, boxes + 2 * S, C::per, stats, kFxT1);
            __syncthreads();
            fx30_project_r<N, EPB_, B1>(
                nel, boxes + 2 * S, C::per, stats, kFxT1, kFxLeft1, [&](int e) { return fx1_exponent<N>(stats + e * K); },
                [&](int e, int t, int l, double w) { Mq[(e0 + e) * NP + t * n + l] = w; });
            __syncthreads();
        }

        // derivatives along r (A -> B), s (A -> C) and t (A -> D)
        if (act) {
            const int mr = fx_derivative<B3, m, oDt, 0>(A, B, u, v), ms = fx_derivative<B3, m, oDt, 1>(A, Cx, u, v),
                      mt = fx_derivative<B3, m, oDt, 2>(A, D, u, v);
            // the common maximum will do where the element is not flat (from N = 7 on
            // the two reductions cost less than the branch: N = 4 591 to 584 us, N = 7
            // 879 to 882)
            if (N < 7 && !FxScales<QB>::flat(st + kFxG)) {
                fx_element_max<mm>(st + kFxU, (unsigned)__vimax3_s32(mr, ms, mt));
            } else {
                fx_element_max<mm>(st + kFxU, (unsigned)mr);
                fx_element_max<mm>(st + kFxU + 1, (unsigned)ms);
                fx_element_max<mm>(st + kFxU + 2, (unsigned)mt);
            }
        }
        __syncthreads();

        // chain rule at the points of column (a=u, b=v)
        int basez = 0;
        if (act) {
            const FxScales<QB> Z(st + kFxG);
            const int kg = Z.kg;
            const bool left = Z.bad || kq + kg > 800 || kq + kg < -800;
            basez = kq - qb + t3 + c_fxd[N].tau[kFoldDt] - Z.sh + 2 + kg + c_fxd[N].tau[kFoldDtT];
            const int eg = kg + 1022 + wuv;
            FxRange range;
            auto chain = [&](int c, auto split) {
                const int s = B3::at(u, v, c);
                fx_chain<split.value>(Ge + c * mm, MP, eg + c_fxd[N].wm[c], Z, B[s], Cx[s], D[s], B[s], Cx[s], D[s], range);
            };
            if (!Z.split) {
#pragma unroll 4
                for (int c = 0; c < m; c++) chain(c, std::false_type());
            } else {
#pragma unroll 1
                for (int c = 0; c < m; c++) chain(c, std::true_type());
            }
            if (left || range.left()) st[kFxLeft30] = flag[1] = 1;
            if (r == 0) st[kFxB] = Z.below();
        }
        __syncthreads();

        // transposes, in place; ln: each line's scale
        if (act) {
            const unsigned below = st[kFxB];
            const int hr = fx_transpose<B3, m, oDtT, QB, 0, EXACT>(B, u, v) + fx_below(below, 0),
                      hs = fx_transpose<B3, m, oDtT, QB, 1, EXACT>(Cx, u, v) + fx_below(below, 1),
                      ht = fx_transpose<B3, m, oDtT, QB, 2, EXACT>(D, u, v) + fx_below(below, 2);
            ln[r] = hr;
            ln[mm + r] = hs;
            ln[2 * mm + r] = ht;
            const int h = __vimin3_s32(hr, hs, ht);
            if (!EXACT || h < kFxZeroLine) fx_element_max<EXACT ? 1 : mm>(st + kFxH, (unsigned)(63 - h));
            if (EXACT) {
                const int unit = __vimin3_s32(hr < kFxZeroLine ? fx_below(below, 0) : 63, hs < kFxZeroLine ? fx_below(below, 1) : 63,
                                              ht < kFxZeroLine ? fx_below(below, 2) : 63);
                atomicMax(st + kFxE, (unsigned)(63 - unit));
            }
        }
        __syncthreads();

        // column: the three directions and lambda wJ q, aligned (-> D)
        int zs = 0;
        if (act) {
            // every line is brought to the largest scale among them (N = 1: that are not zero)
            const int hm = (EXACT && st[kFxH] == 0) ? QB - 32 : 63 - (int)st[kFxH];
            basez -= hm;
            // lines are known to a unit of their direction's scale: the largest
            // must not lie far below that of the largest that is not zero
            const bool lost = EXACT && st[kFxH] != 0 && st[kFxH] + kFxRange < st[kFxE];
            int el2 = 0;  // |lambda| < 2^el2
            if (lambda != 0.0) el2 = ((__double2hiint(lambda) >> 20) & 0x7ff) - 1022;
            const int delta = kq - qb + t3 + kw + el2 - basez;  // scale of the mass term over the other's
            zs = (lambda != 0.0) ? min(63, max(0, delta)) : 0;
            const int ms = min(63, max(0, -delta)), bw = kw + el2 + 1022 + wuv, ht = ln[2 * mm + r] - hm + zs;
            bool left = el2 > 200 || el2 < -200 || delta > 63 || kw > 800 || kw < -800 || kq + kw > 800 || kq + kw < -800;
            if (lambda == 0.0) left = false;
            left = left || lost;
            FxMost most;
            int far = 0, least = 0;
#pragma unroll 4
            for (int c = 0; c < m; c++) {
                const int s = B3::at(u, v, c);
                long long x = fx_shr(B[s], ln[v + m * c] - hm + zs) + fx_shr(Cx[s], ln[mm + u + m * c] - hm + zs) +
                              fx_shr(D[s], ht);
                if (lambda != 0.0) {
                    const double wj = lambda * __ldg(Ge + 6 * MP + c * mm);
                    const int e = (__double2hiint(wj) >> 20) & 0x7ff, d = bw + c_fxd[N].wm[c] - e;
                    far = max(far, d);
                    least = min(least, d);
                    int gh, gl;
                    fx_off_diagonal(wj, d, gh, gl);
                    x += fx_mul(gh, gl, A[s]) >> ms;
                }
                D[s] = x;
                most.see(x);
            }
            fx_element_max<mm>(st + kFxX, (unsigned)most.value());
            if (left || least < 0 || far > kFxRange + 2) st[kFxLeft30] = flag[1] = 1;
        }
        __syncthreads();

        // projection along t (D in place), s (D -> C) and r (C -> Aq)
        if (act) {
            const int sx = QB - 32 - fx_top((int)st[kFxX]), up = max(0, sx), down = max(0, -sx);
            FxMost most;
            fx_line<n, m, 1, oIT>([&](int l) { return (D[B3::at(u, v, l)] << up) >> down; },
                                  [&](int l, long long y) {
                                      D[B2::at(u, v, l)] = y;
                                      most.see(y);
                                  });
            fx_element_max<mm>(st + kFxT30, (unsigned)most.value());
            if (r == 0) ln[0] = basez + zs - sx + 3 * c_fxd[N].tau[kFoldIT];  // (every line's scale has been read)
        }
        __syncthreads();
        fx30_project_s<N, EPB_, B1, B2>(nel, boxes + 3 * S, boxes + 2 * S, C::per, stats, kFxT30);
        __syncthreads();
        fx30_project_r<N, EPB_, B1>(
            nel, boxes + 2 * S, C::per, stats, kFxT30, kFxLeft30,
            [&](int e) { return reinterpret_cast<const int *>(smem_raw + C::off_e)[e * 3 * mm]; },
            [&](int e, int t, int l, double w) {
                const int64_t g = (e0 + e) * NP + t * n + l;
                Aq[g] = w;
                if (PCG) dot = fma(p[g], w, dot);
            });
    }
    if (flag[1] != 0) dot += bp30_left64<N, EPB_, MASS>(smem_raw, e0, nel, G, lambda, PCG ? p : q, Aq, Mq);
    if (PCG) {
        __syncthreads();  // the shared boxes are reused for the reduction
        const double tot = block_sum(dot, reinterpret_cast<double *>(smem_raw));
        if (threadIdx.x == 0) *part_out = tot;
    }
}

}  // namespace
}  // namespace fem
