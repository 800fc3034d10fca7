// BP3.5 in FP64 with its arithmetic on the integer multiply-add pipe (fx.cuh),
// shared by the stand-alone kernels (bp35_fx.cu) and the batched persistent
// kernel (batch.cu).
//
// Each element is a block of fixed-point numbers whose scales follow its
// data, phase by phase:
//   1. q, scaled by the element's largest |q|: 60 bits (59 above 10 points);
//   2. derivatives D q, then scaled up by their largest value (for a smooth
//      field they are far below the bound ||D|| max|q|);
//   3. chain rule: the factors without their quadrature weights' powers of
//      two, scaled by the element's largest diagonal factor to 62 bits, times
//      the derivatives; on flat elements a scale for each direction (FxScales);
//   4. transposes, each line scaled up by its own largest value, the weights
//      in the operator (fx.cuh);
//   5. the three directions aligned to the largest scale at a node, summed,
//      converted and rounded to FP64; lambda wJ q in FP64.
// What bounds it: the integer multiply-adds (at N = 7 two thirds of their
// rate, 404 instructions per node of which 99 multiply-adds; HBM at 53 %).
// Measured on 32^3 elements at N = 7: 331 us (50.5 GDOF/s) against 1555 us of
// the FP64 lines, which ran at the FP64 pipe's rate; 3.4 to 4.2 times faster
// at every other degree from 3 on.  The error against quadruple precision on
// jittered elements is 0.5 to 0.96 of the FP64 lines' for random fields (N =
// 11: 1.06, of which the rounding of the operator tables, common to both, is
// 0.9) and 0.2 to 0.8 for smooth ones.
//
// An element whose values do not share a scale is computed in FP64 instead
// (bp35_element64), by the same block: non-finite or extreme values,
// a node whose result is made of values all far smaller than the element's
// largest (in FP64 it keeps digits that the element's scale cuts off), a
// point whose factors are far smaller than the element's largest, or an
// off-diagonal factor above every diagonal one (G not positive definite).  At
// two and three points a line, where FP64 takes the derivative of a constant
// (at two of any line) without an error, also a node whose lines hold far less
// than the scale of the directions that reach it.
// The choice is made element by element, so a result does not depend on the
// other elements of the block.  Of a smooth field that vanishes on the faces
// of a box, the elements along the box's edges go this way (0.6 % of 32^3
// elements, 5 % of 13^3); of random fields none.
#pragma once

#include "bp35_body.cuh"  // Bp35Layout
#include "fx.cuh"
#include "fx_point.cuh"

namespace fem {
namespace {

template <int N, int EPB_>
struct Fx35Layout : Bp35Layout<double, N, EPB_> {
    using L = Bp35Layout<double, N, EPB_>;
    // per element: max q; max Grr, Gss, Gtt; max derivative along r, s, t; left out; values below a unit;
    // the directions' scales (fx_below)
    static constexpr int kStats = 10;
    // boxes, then a word per line, then the statistics
    static constexpr int off_e = L::bytes;
    static constexpr int off_s = off_e + EPB_ * 3 * L::nn * 4;
    static constexpr int fx_bytes = off_s + EPB_ * kStats * 4;
    static constexpr int smem = fx_bytes > L::smem ? fx_bytes : L::smem;
};

// Algorithm 4 in FP64 on one element by the whole block, sizes at run time
// (fx_line64): q, G and Aq at the element, smem at least 3 n^3 doubles (rows
// of n, or n + 1 for even n, against bank conflicts).  Returns the thread's
// share of q . Aq.
__device__ __noinline__ double bp35_element64(double *smem, int n, int oD, int oDT, const double *G, double lambda,
                                              const double *q, double *Aq) {
    const int nn = n * n, NP = nn * n, sj = n | 1, sk = sj * n, size = sk * n;
    double *sQ = smem, *sR = sQ + size, *sS = sR + size;
    __syncthreads();  // the shared memory is free
    for (int t = threadIdx.x; t < NP; t += blockDim.x) sQ[t % n + sj * ((t / n) % n) + sk * (t / nn)] = q[t];
    __syncthreads();
    const int r = threadIdx.x, u = r % n, v = r / n;
    double ut[kMaxN + 1], acc[kMaxN + 1], dot = 0.0;
    if (r < nn) {
        fx_line64(sQ + sj * u + sk * v, 1, sR + sj * u + sk * v, 1, n, n, -1, oD);
        fx_line64(sQ + u + sk * v, sj, sS + u + sk * v, sj, n, n, -1, oD);
        fx_line64(sQ + u + sj * v, sk, ut, 1, n, n, -1, oD);
    }
    __syncthreads();
    if (r < nn) {
        for (int k = 0; k < n; k++) {
            const int s = u + sj * v + sk * k;
            const double *g = G + r + k * nn, qr = sR[s], qs = sS[s], qt = ut[k];
            sR[s] = g[0] * qr + g[NP] * qs + g[2 * NP] * qt;
            sS[s] = g[NP] * qr + g[3 * NP] * qs + g[4 * NP] * qt;
            ut[k] = g[2 * NP] * qr + g[4 * NP] * qs + g[5 * NP] * qt;
        }
        fx_line64(ut, 1, acc, 1, n, n, -1, oDT);
    }
    __syncthreads();
    if (r < nn) {
        fx_line64(sR + sj * u + sk * v, 1, sR + sj * u + sk * v, 1, n, n, -1, oDT);
        fx_line64(sS + u + sk * v, sj, sS + u + sk * v, sj, n, n, -1, oDT);
    }
    __syncthreads();
    if (r < nn) {
        for (int k = 0; k < n; k++) {
            const int s = u + sj * v + sk * k;
            double w = acc[k];
            if (lambda != 0.0) w = fma(lambda, G[6 * NP + r + k * nn] * sQ[s], w);
            w = w + sR[s] + sS[s];
            Aq[r + k * nn] = w;
            dot = fma(sQ[s], w, dot);
        }
    }
    return dot;
}

// Whether node (i, j, k), none of whose lines reaches the element's scale, is
// held to it all the same: by the off-diagonal factors, through the lines
// that cross its own (a node on an edge of a field that vanishes on two
// faces), or because everything that enters its result is zero.  ln: largest
// high word of each r-, s- and t-line (0: all zeros; with `tiny`, possibly
// values below a unit); G: the element's factors.
__device__ __noinline__ bool fx35_held(const int *ln, const double *G, int n, int i, int j, int k, const int *wn, int kg,
                                       int need, bool tiny) {
    const int nn = n * n, NP = nn * n;
    bool any = tiny || (ln[j + n * k] | ln[nn + i + n * k] | ln[2 * nn + i + n * j]) != 0;
    // a line and the factor that multiplies its derivative at point (a, b, c)
    auto held = [&](int line, int h, int a, int b, int c) {
        const int e = (__double2hiint(__ldg(G + h * NP + a + n * b + nn * c)) >> 20) & 0x7ff;
        if (line == 0 || e == 0) return false;
        any = true;
        return fx_top(line) + e - 1022 - wn[a] - wn[b] - wn[c] - kg >= need;
    };
    for (int l = 0; l < n; l++) {
        if (held(ln[nn + l + n * k], 1, l, j, k) || held(ln[2 * nn + l + n * j], 2, l, j, k) ||
            held(ln[l + n * k], 1, i, l, k) || held(ln[2 * nn + i + n * l], 4, i, l, k) ||
            held(ln[j + n * l], 2, i, j, l) || held(ln[nn + i + n * l], 4, i, j, l))
            return true;
    }
    return !any;
}

// BP3.5 of elements [e0, e0 + nel) by the whole block (blockDim.x >=
// Layout::threads), as bp35_block.
template <int N, int EPB_, bool PCG>
__device__ __forceinline__ void bp35_fx_block(unsigned char *smem_raw, int64_t e0, int nel,
                                              const double *__restrict__ G, double lambda, const double *__restrict__ q,
                                              double *__restrict__ Aq, const double *__restrict__ z, double *p,
                                              const double *__restrict__ beta, double *__restrict__ part_out) {
    using C = Fx35Layout<N, EPB_>;
    using B = typename C::B;
    constexpr int n = C::n, nn = C::nn, NP = C::NP, QB = fx_bits35(N), K = C::kStats;
    constexpr bool EXACT = n <= 3;  // FP64 lines may make no error
    constexpr int UC = 4;  // nodes of a column taken at a time (whole columns spill)
    constexpr int oD = fold_offset(N, kFoldD), oDT = fold_offset(N, kFoldDT);
    const int el = threadIdx.x / nn, r = threadIdx.x - el * nn;
    const int u = r % n, v = r / n;
    const bool act = el < nel;
    long long *box = reinterpret_cast<long long *>(smem_raw) + el * 3 * B::size;  // three boxes
    int *ln = reinterpret_cast<int *>(smem_raw + C::off_e) + el * 3 * nn;         // a word per line
    unsigned *stats = reinterpret_cast<unsigned *>(smem_raw + C::off_s), *st = stats + el * K;
    if (threadIdx.x == 0) prefetch_l2(G + e0 * 7 * NP, (long long)nel * 7 * NP * 8);
    for (int t = threadIdx.x; t < EPB_ * K; t += blockDim.x) stats[t] = 0;
    __syncthreads();

    // the element's largest field value
    const double *Ge = G + (e0 + el) * 7 * NP + r;
    const int wuv = act ? c_fxd[N].wn[u] + c_fxd[N].wn[v] : 0;
    double qv[n];
    if (act) {
        const int64_t g0 = (e0 + el) * NP + r;
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
        unsigned m = 0;
#pragma unroll
        for (int k = 0; k < n; k++) m = max(m, (unsigned)fx_abs_hi(qv[k]));
        fx_element_max<nn>(st + 0, m);
    }
    __syncthreads();

    // scale: |q| < 2^kq
    constexpr int qb = QB - 1;
    int kq = 0;
    if (act) {
        const unsigned qm = st[0];
        const int eq = (int)(qm >> 20);
        kq = qm ? eq - 1022 : 0;
        bool bad = (qm != 0 && eq < 64) || eq == 0x7ff;
        if (qm == 0) {  // zeros, or values below 2^-1042
#pragma unroll
            for (int k = 0; k < n; k++) bad = bad || __double2loint(qv[k]) != 0;
        }
        if (bad) st[7] = 1;
        int most = 0;  // largest shift of a value that is not zero
#pragma unroll
        for (int k = 0; k < n; k++) {
            const int sq = kq + 1022 - (int)((__double2hiint(qv[k]) >> 20) & 0x7ff);
            if ((fx_abs_hi(qv[k]) | __double2loint(qv[k])) != 0) most = max(most, sq);
            box[B::at(u, v, k)] = fx_from_double<qb>(qv[k], sq);
        }
        if (most >= qb) st[8] = 1;
    }
    __syncthreads();

    // derivatives along r and s to boxes 1 and 2, then along t in place in
    // box 0; ln: each line's largest value
    if (act) {
        const int mr = fx_derivative<B, n, oD, 0, true>(box, box + B::size, u, v, ln + r),
                  ms = fx_derivative<B, n, oD, 1, true>(box, box + 2 * B::size, u, v, ln + nn + r);
        fx_element_max<nn>(st + 4, (unsigned)mr);
        fx_element_max<nn>(st + 5, (unsigned)ms);
    }
    __syncthreads();
    if (act) {
        fx_element_max<nn>(st + 6, (unsigned)fx_derivative<B, n, oD, 2, true>(box, box, u, v, ln + 2 * nn + r));
        // the diagonal factors' largest exponents, without the weights
        // (prefetched into L2 when the block began)
        int gm[3] = {0, 0, 0};
        const int *Gi = reinterpret_cast<const int *>(Ge) + 1;  // high words
#pragma unroll(UC)
        for (int k = 0; k < n; k++) {
            const int w = c_fxd[N].wn[k] << 20;
#pragma unroll
            for (int h = 0; h < 3; h++) gm[h] = max(gm[h], __ldg(Gi + 2 * ((h == 0 ? 0 : 1 + 2 * h) * NP + k * nn)) - w);
        }
#pragma unroll
        for (int h = 0; h < 3; h++) fx_element_max<nn>(st + 1 + h, (unsigned)(gm[h] - (wuv << 20)));
    }
    __syncthreads();

    // chain rule at the nodes of column (i=u, j=v)
    int base = 0;
    if (act) {
        const FxScales<QB> S(st + 1);
        const int kg = S.kg;
        bool bad = S.bad || kq + kg > 800 || kq + kg < -800;
        // a node is held to the element's scale by its largest line; kd: diagonal factors without weights < 2^kd
        const int most = (int)(max(st[1], max(st[2], st[3])) >> 20);
        auto kd = [&](int d) { return (int)(st[1 + d] >> 20) - most; };
        const int need = qb - 32 - kFxRange;  // bits of a line's high word, with its factor at the largest
        const int lt = ln[2 * nn + r];
        if (fx_top(lt) + kd(2) < need) {
#pragma unroll 1
            for (int k = 0; k < n; k++)
                if (fx_top(ln[v + n * k]) + kd(0) < need && fx_top(ln[nn + u + n * k]) + kd(1) < need)
                    bad = bad || !fx35_held(ln, G + (e0 + el) * 7 * NP, n, u, v, k, c_fxd[N].wn, most - 1022, need,
                                            st[8] != 0);
        }
        base = kq - qb + c_fxd[N].tau[kFoldD] - S.sh + 2 + kg + c_fxd[N].tau[kFoldDT];
        const int eg = kg + 1022 + wuv;
        FxRange range;
        auto chain = [&](int k, auto split) {
            const int s = B::at(u, v, k);
            long long *rr = box + B::size + s, *ss = rr + B::size, *tt = box + s;
            fx_chain<split.value>(Ge + k * nn, NP, eg + c_fxd[N].wn[k], S, *rr, *ss, *tt, *rr, *ss, *tt, range);
        };
        if (!S.split) {
#pragma unroll(UC)
            for (int k = 0; k < n; k++) chain(k, std::false_type());
        } else {
#pragma unroll 1
            for (int k = 0; k < n; k++) chain(k, std::true_type());
        }
        if (bad || range.left()) st[7] = 1;
        if (r == 0) st[9] = S.below();
    }
    __syncthreads();

    // transposes, in place; ln: each line's exponent
    if (act) {
        ln[r] = -fx_transpose<B, n, oDT, QB, 0, EXACT>(box + B::size, u, v) - fx_below(st[9], 0);
        ln[nn + r] = -fx_transpose<B, n, oDT, QB, 1, EXACT>(box + 2 * B::size, u, v) - fx_below(st[9], 1);
        ln[2 * nn + r] = -fx_transpose<B, n, oDT, QB, 2, EXACT>(box, u, v) - fx_below(st[9], 2);
    }
    __syncthreads();

    // a node's lines are known to a unit of their directions' scale: its
    // largest must not lie far below that of the largest that is not zero
    if constexpr (EXACT) {
        if (act) {
            const unsigned below = st[9];
            const int et = ln[2 * nn + r];
#pragma unroll
            for (int k = 0; k < n; k++) {
                const int a = ln[v + n * k], b = ln[nn + u + n * k];
                const int unit = __vimax3_s32(a > -kFxZeroLine ? -fx_below(below, 0) : -kFxZeroLine,
                                              b > -kFxZeroLine ? -fx_below(below, 1) : -kFxZeroLine,
                                              et > -kFxZeroLine ? -fx_below(below, 2) : -kFxZeroLine);
                if (unit > -kFxZeroLine && __vimax3_s32(et, a, b) < unit - kFxRange) st[7] = 1;
            }
        }
        __syncthreads();
    }

    double dot = 0.0;  // p . Ap of the thread's column
    if (act && st[7] == 0) {
        const int64_t g0 = (e0 + el) * NP + r;
        const double *qe = PCG ? p : q;
        const int et = ln[2 * nn + r];
#pragma unroll(UC)
        for (int k = 0; k < n; k++) {
            const int s = B::at(u, v, k);
            const int a = ln[v + n * k], b = ln[nn + u + n * k], d = __vimax3_s32(et, a, b);
            const long long sum =
                fx_shr(box[s], d - et) + fx_shr(box[B::size + s], d - a) + fx_shr(box[2 * B::size + s], d - b);
            double w = fx_to_double(sum, base + d + wuv + c_fxd[N].wn[k]);
            const double qk = qe[g0 + k * nn];
            if (lambda != 0.0) w = fma(lambda, __ldg(Ge + 6 * NP + k * nn) * qk, w);
            Aq[g0 + k * nn] = w;
            if (PCG) dot = fma(qk, w, dot);
        }
    }
    for (int e = 0; e < nel; e++)
        if (stats[e * K + 7] != 0) {  // the same for every thread
            const double d = bp35_element64(reinterpret_cast<double *>(smem_raw), n, oD, oDT, G + (e0 + e) * 7 * NP,
                                            lambda, (PCG ? p : q) + (e0 + e) * NP, Aq + (e0 + e) * NP);
            if (PCG) dot += d;
        }
    if (PCG) {
        __syncthreads();  // the shared boxes are reused for the reduction
        const double tot = block_sum(dot, reinterpret_cast<double *>(smem_raw));
        if (threadIdx.x == 0) *part_out = tot;
    }
}

}  // namespace
}  // namespace fem
