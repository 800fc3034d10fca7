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
// rate, 99 of about 410 instructions per node; HBM at 52 %).
// Measured on 32^3 elements at N = 7: 342 us (49.0 GDOF/s) against 1555 us of
// the FP64 lines, which ran at the FP64 pipe's rate; 3.0 to 4.0 times faster
// at every other degree from 3 on.  The error against quadruple precision on
// jittered elements is 0.21 to 0.71 of the FP64 lines' for random fields, 0.49
// to 0.74 for smooth ones.
//
// An element whose values do not share a scale is computed in FP64 instead
// (bp35_left64), by the same block: non-finite or extreme values, a node whose
// result is made of values all far smaller than the element's largest (in FP64
// it keeps digits that the element's scale cuts off), a point whose factors are
// far smaller than the element's largest, directions further apart than
// kFxApart, or an off-diagonal factor above every diagonal one (G not positive
// definite).  Element by element, so a result does not depend on the other
// elements of the block.  What the field or a factor's sign tells, before the
// contractions; the rest when the factors are known.  A mesh of such elements
// takes 0.85 to 1.05 of the FP64 kernel's time.  Of a smooth field that
// vanishes on the faces of a box, the elements along the box's edges go this
// way (0.6 % of 32^3 elements, 5 % of 13^3); of random fields none.
#pragma once

#include "bp35_body.cuh"  // Bp35Layout
#include "fx.cuh"
#include "fx_point.cuh"

namespace fem {
namespace {

// Slots of an element's statistics: the largest q, Grr, Gss, Gtt and
// derivatives along r, s, t (FxScales), whether the element is left to FP64,
// whether it holds values below a unit, the directions' scales (fx_below), the
// largest q of each face.
enum { kFx35Q = 0, kFx35G = 1, kFx35Left = 7, kFx35Tiny = 8, kFx35B = 9, kFx35F = 10, kFx35Stats = 16 };

// At two and three points a line BP3.5 stays in FP64: its derivatives of a
// constant line (at two points of any line) have no error there, so a node far
// below its element's largest keeps digits that one scale cuts off, and of a
// smooth field so many elements hold such nodes that the fixed point gained
// nothing (N = 1, 2 on a product of sines: 46 and 78 us against 40 and 78).
__host__ __device__ constexpr bool fx35_fixed(int N) { return N >= 3; }

template <int N, int EPB_>
struct Fx35Layout : Bp35Layout<double, N, EPB_> {
    using L = Bp35Layout<double, N, EPB_>;
    static constexpr int kStats = kFx35Stats;
    // boxes, then a word per line, the statistics and three flags of the block: an
    // element is on the fixed-point path; one is left to FP64; one has a small corner
    static constexpr int off_e = L::bytes;
    static constexpr int off_s = off_e + EPB_ * 3 * L::nn * 4;
    static constexpr int off_b = off_s + EPB_ * kStats * 4;  // the block's flags
    static constexpr int fx_bytes = off_b + 12;
    static constexpr int smem = fx_bytes > L::smem ? fx_bytes : L::smem;
};

// Algorithm 4 in FP64 on the block's elements [e0, e0 + nel) for which on(el)
// holds, all of them at once, a line per thread as on the fixed-point path and
// in its boxes.  Returns the thread's share of q . Aq.
template <int N, int EPB_, class F>
__device__ __forceinline__ double bp35_lines64(unsigned char *smem_raw, int64_t e0, int nel, const double *G,
                                               double lambda, const double *q, double *Aq, F &&on) {
    using C = Fx35Layout<N, EPB_>;
    using B = typename C::B;
    constexpr int n = C::n, nn = C::nn, NP = C::NP;
    constexpr int oD = fold_offset(N, kFoldD), oDT = fold_offset(N, kFoldDT);
    const int el = threadIdx.x / nn, r = threadIdx.x - el * nn;
    const int u = r % n, v = r / n;
    const bool act = el < nel && on(el);
    const int64_t g0 = (e0 + el) * NP + r;
    double *box = reinterpret_cast<double *>(smem_raw) + el * 3 * B::size, *bs = box + B::size, *bt = bs + B::size;
    // the thread's line of direction d from one box to another, or in place; the
    // directions take turns in one loop (side by side they spilled)
    auto line = [&](auto off, int d, const double *from, double *to) {
        const int step = d == 0 ? 1 : d == 1 ? B::sj : B::sk,
                  at = d == 0 ? B::at(0, u, v) : d == 1 ? B::at(u, 0, v) : B::at(u, v, 0);
        double x[n];
#pragma unroll
        for (int l = 0; l < n; l++) x[l] = from[at + l * step];
        fx_line64<n, n, -1, off.value>(x, [&](int l, double y) { to[at + l * step] = y; });
    };
    using D = std::integral_constant<int, oD>;
    using DT = std::integral_constant<int, oDT>;
    __syncthreads();  // the shared memory is free
    if (act) {
#pragma unroll
        for (int k = 0; k < n; k++) box[B::at(u, v, k)] = q[g0 + k * nn];
    }
    __syncthreads();
    // derivatives along t and s to boxes 2 and 1, then along r in place in box 0
#pragma unroll 1
    for (int d = 2; d >= 0; d--) {
        if (d == 0) __syncthreads();
        if (act) line(D(), d, box, box + d * B::size);
    }
    __syncthreads();
    if (act) {
        const double *g = G + (e0 + el) * 7 * NP + r;
#pragma unroll 2
        for (int k = 0; k < n; k++, g += nn) {
            const int s = B::at(u, v, k);
            const double qr = box[s], qs = bs[s], qt = bt[s], g1 = __ldg(g + NP), g2 = __ldg(g + 2 * NP),
                         g4 = __ldg(g + 4 * NP);
            box[s] = fx_dot64(__ldg(g), qr, g1, qs, g2, qt);
            bs[s] = fx_dot64(g1, qr, __ldg(g + 3 * NP), qs, g4, qt);
            bt[s] = fx_dot64(g2, qr, g4, qs, __ldg(g + 5 * NP), qt);
        }
    }
    __syncthreads();
    if (act) {
#pragma unroll 1
        for (int d = 0; d < 3; d++) line(DT(), d, box + d * B::size, box + d * B::size);
    }
    __syncthreads();
    double dot = 0.0;
    if (act) {
#pragma unroll 2
        for (int k = 0; k < n; k++) {
            const int s = B::at(u, v, k);
            const double qk = q[g0 + k * nn];
            double w = bt[s];
            if (lambda != 0.0) w = fma(lambda, __dmul_rn(__ldg(G + (e0 + el) * 7 * NP + 6 * NP + r + k * nn), qk), w);
            w = w + box[s] + bs[s];
            Aq[g0 + k * nn] = w;
            dot = fma(qk, w, dot);
        }
    }
    return dot;
}

// The same as a function of its own, for the elements that the fixed-point path
// leaves out (stats: their flags), so that its registers are not the fast path's.
template <int N, int EPB_>
__device__ __noinline__ double bp35_left64(unsigned char *smem_raw, int64_t e0, int nel, const double *G, double lambda,
                                           const double *q, double *Aq) {
    using C = Fx35Layout<N, EPB_>;
    const unsigned *stats = reinterpret_cast<const unsigned *>(smem_raw + C::off_s);
    return bp35_lines64<N, EPB_>(smem_raw, e0, nel, G, lambda, q, Aq,
                                 [&](int el) { return stats[el * C::kStats + kFx35Left] != 0; });
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

// Leaves out elements with a corner whose three faces hold values far below the
// element's largest only: it is not held to the element's scale (fx35_held reads
// its faces), which this tells before the contractions, from the scaled field.
// (Fields that decay across an element are made of such elements.)  Returns
// whether elements are left on the fixed-point path.
template <int N, int EPB_>
__device__ __noinline__ bool fx35_corners(unsigned char *smem_raw, int nel) {
    using C = Fx35Layout<N, EPB_>;
    using B = typename C::B;
    constexpr int n = C::n, nn = C::nn, need = fx_bits35(N) - 1 - 32 - kFxRange;
    const int el = threadIdx.x / nn, r = threadIdx.x - el * nn, u = r % n, v = r / n;
    unsigned *stats = reinterpret_cast<unsigned *>(smem_raw + C::off_s), *st = stats + el * C::kStats;
    if (el < nel) {
        const long long *box = reinterpret_cast<const long long *>(smem_raw) + el * 3 * B::size;
        auto value = [&](int k) {
            const int h = (int)(box[B::at(u, v, k)] >> 32);
            return (unsigned)max(h, ~h);
        };
        unsigned m = 0;
        for (int k = 0; k < n; k++) m = max(m, value(k));
        if (u == 0) atomicMax(st + kFx35F, m);
        if (u == n - 1) atomicMax(st + kFx35F + 1, m);
        if (v == 0) atomicMax(st + kFx35F + 2, m);
        if (v == n - 1) atomicMax(st + kFx35F + 3, m);
        atomicMax(st + kFx35F + 4, value(0));
        atomicMax(st + kFx35F + 5, value(n - 1));
    }
    __syncthreads();
    if (el < nel && r == 0) {
        const unsigned *f = st + kFx35F;
        const unsigned least = max(max(min(f[0], f[1]), min(f[2], f[3])), min(f[4], f[5]));
        if (least != 0 && fx_top((int)least) < need) {
            st[kFx35Left] = 1;
            reinterpret_cast<volatile unsigned *>(smem_raw + C::off_b)[1] = 1;
        }
    }
    __syncthreads();
    bool some = false;
    for (int e = 0; e < nel; e++) some = some || stats[e * C::kStats + kFx35Left] == 0;
    return some;
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
    // nodes of a column taken at a time: whole columns spill; five where they leave
    // less over (32^3 elements and more: N = 6 385 to 371 us, N = 8 404 to 398, N = 7
    // 349 to 368)
    constexpr int UC = (N == 4 || N == 6 || N == 8 || N == 9) ? 5 : 4;
    constexpr int oD = fold_offset(N, kFoldD), oDT = fold_offset(N, kFoldDT);
    const int el = threadIdx.x / nn, r = threadIdx.x - el * nn;
    const int u = r % n, v = r / n;
    const bool act = el < nel;
    long long *box = reinterpret_cast<long long *>(smem_raw) + el * 3 * B::size;  // three boxes
    int *ln = reinterpret_cast<int *>(smem_raw + C::off_e) + el * 3 * nn;         // a word per line
    unsigned *stats = reinterpret_cast<unsigned *>(smem_raw + C::off_s), *st = stats + el * K;
    if (threadIdx.x == 0) prefetch_l2(G + e0 * 7 * NP, (long long)nel * 7 * NP * 8);
    if constexpr (!fx35_fixed(N)) {
        if (PCG && act) {
            const int64_t g0 = (e0 + el) * NP + r;
            const double bt = *beta;
#pragma unroll
            for (int k = 0; k < n; k++) {
                const int64_t g = g0 + k * nn;
                p[g] = (bt == 0.0) ? z[g] : fma(bt, p[g], z[g]);
            }
        }
        const double d = bp35_lines64<N, EPB_>(smem_raw, e0, nel, G, lambda, PCG ? p : q, Aq, [](int) { return true; });
        if (PCG) {
            __syncthreads();  // the shared boxes are reused for the reduction
            const double tot = block_sum(d, reinterpret_cast<double *>(smem_raw));
            if (threadIdx.x == 0) *part_out = tot;
        }
        return;
    }
    volatile unsigned *flag = reinterpret_cast<volatile unsigned *>(smem_raw + C::off_b);
    for (int t = threadIdx.x; t < EPB_ * K + 3; t += blockDim.x) stats[t] = 0;  // (the flags lie behind them)
    __syncthreads();

    // the element's largest field value
    const double *Ge = G + (e0 + el) * 7 * NP + r;
    const int wuv = act ? c_fxd[N].wn[u] + c_fxd[N].wn[v] : 0;
    double qv[n];
    int sign = 0;  // of the element's first factor, read ahead (a left-handed mesh has them all negative)
    if (act) {
        const int64_t g0 = (e0 + el) * NP + r;
        if (r == 0) sign = __ldg(reinterpret_cast<const int *>(Ge) + 1);
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
        fx_element_max<nn>(st + kFx35Q, m);
    }
    __syncthreads();

    // scale: |q| < 2^kq
    constexpr int qb = QB - 1;
    int kq = 0;
    if (act) {
        const unsigned qm = st[kFx35Q];
        const int eq = (int)(qm >> 20);
        kq = qm ? eq - 1022 : 0;
        bool bad = (qm != 0 && eq < 64) || eq == 0x7ff;
        if (qm == 0) {  // zeros, or values below 2^-1042
#pragma unroll
            for (int k = 0; k < n; k++) bad = bad || __double2loint(qv[k]) != 0;
        }
        bad = bad || sign < 0;
        if (bad) st[kFx35Left] = 1;
        if (bad) flag[1] = 1;
        if (!bad && r == 0) flag[0] = 1;
        int most = 0;  // largest shift of a value that is not zero
#pragma unroll
        for (int k = 0; k < n; k++) {
            const int sq = kq + 1022 - (int)((__double2hiint(qv[k]) >> 20) & 0x7ff);
            if ((fx_abs_hi(qv[k]) | __double2loint(qv[k])) != 0) most = max(most, sq);
            box[B::at(u, v, k)] = fx_from_double<qb>(qv[k], sq);
        }
        if (most >= qb) st[kFx35Tiny] = 1;
        if ((u == 0 || u == n - 1) && (v == 0 || v == n - 1)) {  // a corner far below the element's largest value
            const int far = eq - 2 * kFxRange;
            if ((fx_abs_hi(qv[0]) >> 20) < far || (fx_abs_hi(qv[n - 1]) >> 20) < far) flag[2] = 1;
        }
    }
    __syncthreads();
    double dot = 0.0;  // p . Ap of the thread's column
    bool go = flag[0] != 0;
    if (flag[2] != 0 && go) go = fx35_corners<N, EPB_>(smem_raw, nel);
    if (go) {
        // derivatives along r and s to boxes 1 and 2, then along t in place in
        // box 0; ln: each line's largest value
        if (act) {
            const int mr = fx_derivative<B, n, oD, 0, true>(box, box + B::size, u, v, ln + r),
                      ms = fx_derivative<B, n, oD, 1, true>(box, box + 2 * B::size, u, v, ln + nn + r);
            fx_element_max<nn>(st + kFx35G + 3, (unsigned)mr);
            fx_element_max<nn>(st + kFx35G + 4, (unsigned)ms);
        }
        __syncthreads();
        if (act) {
            const int mt = fx_derivative<B, n, oD, 2, true>(box, box, u, v, ln + 2 * nn + r);
            fx_element_max<nn>(st + kFx35G + 5, (unsigned)mt);
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
            for (int h = 0; h < 3; h++) fx_element_max<nn>(st + kFx35G + h, (unsigned)(gm[h] - (wuv << 20)));
        }
        __syncthreads();

        // chain rule at the nodes of column (i=u, j=v)
        int base = 0;
        if (act) {
            const FxScales<QB> S(st + kFx35G);
            const int kg = S.kg;
            const bool bad = S.bad || kq + kg > 800 || kq + kg < -800;
            // a node is held to the element's scale by its largest line; kd: diagonal factors without weights < 2^kd
            const int most = (int)(max(st[kFx35G], max(st[kFx35G + 1], st[kFx35G + 2])) >> 20);
            auto kd = [&](int d) { return (int)(st[kFx35G + d] >> 20) - most; };
            const int need = qb - 32 - kFxRange;  // bits of a line's high word, with its factor at the largest
            const int lt = ln[2 * nn + r];
            if (fx_top(lt) + kd(2) < need) {
                volatile unsigned *left = st + kFx35Left;  // (one node that is not held leaves the element out)
#pragma unroll 1
                for (int k = 0; k < n && *left == 0; k++)
                    if (fx_top(ln[v + n * k]) + kd(0) < need && fx_top(ln[nn + u + n * k]) + kd(1) < need &&
                        !fx35_held(ln, G + (e0 + el) * 7 * NP, n, u, v, k, c_fxd[N].wn, most - 1022, need,
                                   st[kFx35Tiny] != 0))
                        *left = flag[1] = 1;
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
            if (bad || range.left()) st[kFx35Left] = flag[1] = 1;
            if (r == 0) st[kFx35B] = S.below();
        }
        __syncthreads();

        // transposes, in place; ln: each line's exponent
        const bool on = act && st[kFx35Left] == 0;
        if (on) {
            ln[r] = -fx_transpose<B, n, oDT, QB, 0>(box + B::size, u, v) - fx_below(st[kFx35B], 0);
            ln[nn + r] = -fx_transpose<B, n, oDT, QB, 1>(box + 2 * B::size, u, v) - fx_below(st[kFx35B], 1);
            ln[2 * nn + r] = -fx_transpose<B, n, oDT, QB, 2>(box, u, v) - fx_below(st[kFx35B], 2);
        }
        __syncthreads();

        if (on) {
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
    }
    if (flag[1] != 0) dot += bp35_left64<N, EPB_>(smem_raw, e0, nel, G, lambda, PCG ? p : q, Aq);
    if (PCG) {
        __syncthreads();  // the shared boxes are reused for the reduction
        const double tot = block_sum(dot, reinterpret_cast<double *>(smem_raw));
        if (threadIdx.x == 0) *part_out = tot;
    }
}

}  // namespace
}  // namespace fem
