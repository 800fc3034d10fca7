// Geometric factors of trilinear hexahedra, IEEE FP64 (Section 4):
//   X = dx/d(r,s,t),  |J| = det X,  G = |J| X^{-1} X^{-T},
// each multiplied by the tensor quadrature weight w_a w_b w_c, stored as the
// planes Grr, Grs, Grt, Gss, Gst, Gtt, wJ (BP3.5 at GLL nodes, BP3.0 at
// Gauss points) or wJ alone (BP1.0 at Gauss points).
//
// GB300 design.  The columns of X of a trilinear map factor over the tensor
// grid: dx/dr depends on (s, t) only, dx/ds on (r, t) and dx/dt on (r, s), so
// each block first tabulates the three q x q column tables of its element in
// shared memory (O(q^2) work), then every point needs only the cofactor
// vectors C_r = X_s x X_t, C_s = X_t x X_r, C_t = X_r x X_s (the rows of |J|
// X^{-1}), the determinant X_r . C_r and the six products G = C C^T / |J|.
// Stores are coalesced per plane.
//
// In FP64 that is 52 instructions a point at 2 per clock and SM.  The point
// work therefore runs on the integer multiply-add pipe (fx.cuh) in 62-bit
// fixed point, one scale for each of X_r, X_s, X_t of an element; the result
// is converted to FP64 once.  All factors of 32^3 elements at N = 7 (boxes with
// a 10 % jitter): 1322 us against 4186 in FP64; the bound is the integer
// multiply-adds (about 150 a point, half their rate) and the seven conversions
// on the FP64 pipe.  The error against quadruple precision, relative to
// sqrt(G_aa G_bb), is 0.53 to 0.83 of the FP64 kernel's over all planes.
//
// An element for which the scales do not serve is computed in FP64: a component
// of a column far below the column's largest but not zero (a slightly skewed
// element, whose small off-diagonal factors FP64 gives to full relative
// accuracy), nearly parallel columns (kGeoSquare, kGeoDet), a determinant that
// is not positive, extreme or non-finite vertices.  The choice is made element
// by element; the centre's cofactors make it before any point is computed where
// they can.  So the gain depends on the mesh.  Axis-aligned boxes with their
// vertices moved by 10, 5, 3, 2 and 1 % of the spacing leave 4, 13, 31, 61 and
// 99.8 % of their elements to FP64; at N = 7 on 20^3 elements that takes 369,
// 405, 454, 564 and 969 us (FP64 1072), undisturbed or rotated boxes 328, a
// smooth map 601, a left-handed or a strongly sheared mesh 1074.
#define FEM_FX_TABLES
#include "fx.cuh"

namespace fem {
namespace {

template <int qn>
struct GeoCfg {
    static constexpr int QP = qn * qn * qn, qq = qn * qn;
    static constexpr int SD = qq + 4;  // per-thread minima; three scales and what is left to FP64 (eight words)
    static constexpr int PER = pad2(24 + 36 + 9 * qq + SD);  // vertices, map coefficients, tables, minima
    static constexpr int smem_elem = PER * 8;
    // about 256 threads per block: with four resident blocks 1315 us for all
    // factors at N = 7 on 32^3 elements, against 1396 with two of 512
    static constexpr int EPB = pick_epb(qn, smem_elem, 256);
    static constexpr int threads = qq * EPB;
    static constexpr int smem = (4 * pad2(qn) + EPB * PER) * 8;
};

// 1 / d in FP64: an FP32 reciprocal seed refined by two Newton steps
// r <- r + r (1 - d r), each doubling the correct bits (about 22, 44, then
// the full 53).  The seed's conversions between the IEEE binary64 and
// binary32 formats are done on the bit fields with integer operations
// (sign; exponent rebiased from 1023 to 127; the top 23 mantissa bits,
// truncated), so the FP64 pipe (2 per clock per SM) executes only the four
// FMAs.  Falls back to a division when |d| is outside 2^-120..2^121,
// where the seed or its reciprocal would leave the binary32 normal range.
__device__ __forceinline__ double recip(double d) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const unsigned hi = (unsigned)(b >> 32);
    const int ex = (int)((hi >> 20) & 0x7FFu) - 1023;  // unbiased binary64 exponent
    if (ex < -120 || ex > 120) return 1.0 / d;
    const unsigned fb = (hi & 0x80000000u) | ((unsigned)(ex + 127) << 23) | ((hi & 0xFFFFFu) << 3) |
                        (unsigned)((b >> 29) & 0x7u);
    const unsigned rb = __float_as_uint(__frcp_rn(__uint_as_float(fb)));
    const int rex = (int)((rb >> 23) & 0xFFu) - 127;   // unbiased binary32 exponent of the seed
    const unsigned rhi = (rb & 0x80000000u) | ((unsigned)(rex + 1023) << 20) | ((rb & 0x7FFFFFu) >> 3);
    double r = __longlong_as_double((long long)(((unsigned long long)rhi << 32) |
                                                ((unsigned long long)(rb & 0x7u) << 29)));
    double e = fma(-d, r, 1.0);
    r = fma(r, e, r);
    e = fma(-d, r, 1.0);
    return fma(r, e, r);
}

// a b / 2^(64 - k) of values up to 2^62 (the result below 2^63); k <= 3.
template <int k>
__device__ __forceinline__ long long geo_mul(long long a, long long b) {
    const int ah = fx_hi(a), al = fx_lo(a), bh = fx_hi(b), bl = fx_lo(b);
    const long long m = mad_wide(ah, bl, mad_wide(al, bh, 1ll << (31 - k)));
    return (mul_wide(ah, bh) << k) + (m >> (32 - k));
}
// a b - c d over 2^64.
__device__ __forceinline__ long long geo_cross(long long a, long long b, long long c, long long d) {
    return geo_mul<0>(a, b) - geo_mul<0>(c, d);
}
// a . b over 2^(64 - k) of vectors below 2^62, exact to the last unit when
// below 2^63.
template <int k>
__device__ __forceinline__ long long geo_dot(const long long (&a)[3], const long long (&b)[3]) {
    long long h = 0, m = 0;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        const int ah = fx_hi(a[d]), al = fx_lo(a[d]), bh = fx_hi(b[d]), bl = fx_lo(b[d]);
        h = d == 0 ? mul_wide(ah, bh) : mad_wide(ah, bh, h);
        m += mad_wide(ah, bl, mad_wide(al, bh, 1ll << (31 - k))) >> (32 - k);
    }
    return (h << k) + m;
}

// 2^122 / d for 2^61 <= d < 2^62: a binary32 reciprocal seed and two Newton
// steps r <- r + r (1 - d r), to about 2^-57.
__device__ __forceinline__ long long geo_recip(long long d) {
    const float x = __uint_as_float(0x3f000000u | ((unsigned)(d >> 38) & 0x7fffffu));  // d / 2^62
    const unsigned rb = min(__float_as_uint(__frcp_rn(x)), 0x3fffffffu);               // (1, 2)
    long long r = (long long)((rb & 0x7fffffu) | 0x800000u) << 37;
#pragma unroll
    for (int it = 0; it < 2; it++) r += geo_mul<0>(r, ((1ll << 58) - geo_mul<0>(d, r)) << 6);
    return r;
}

// x 2^(62 - k) for |x| < 2^k, as an integer.
__device__ __forceinline__ long long geo_fixed(double x, int k) {
    return fx_from_double<62>(x, k + 1022 - ((__double2hiint(x) >> 20) & 0x7ff));
}

// A component of a column may lie this many bits below the column's largest.
constexpr int kGeoRange = 6;

// What the fixed point needs of a point, with X^ the columns over their scales
// (components below 1): |C^|^2 of each cofactor vector and det X^ at least
// 2^-7.  The cofactors carry 2^-59 of rounding, their squares and products
// 2^-60 and the determinant 2^-58, all absolute, while FP64 rounds each
// product at its own size: where columns are nearly parallel, or several of
// their components are small, FP64 holds more.  Against quadruple precision
// (3000 rotated, sheared and skewed elements) the fixed point's error is 0.5
// to 0.8 of FP64's above these limits, and passes it below |C^|^2 = 2^-10
// and det = 2^-7.
constexpr int kGeoSquare = 60 - 7, kGeoDet = 59 - 7;  // of a square (over 2^60), a determinant (over 2^59)

// x 2^-k in binary32 for |x| < 2^k (0 below 2^(k-126)), by the bit fields.
__device__ __forceinline__ float geo_float(double x, int k) {
    const int hi = __double2hiint(x), e = ((hi >> 20) & 0x7ff) - 1023 - k + 127;
    const unsigned m = ((unsigned)hi & 0x80000000u) | (unsigned)e << 23 | ((unsigned)hi & 0xfffffu) << 3 |
                       (unsigned)__double2loint(x) >> 29;
    return e > 0 ? __uint_as_float(m) : 0.0f;
}

// kind: 1 = wJ only, 2 and 3 = 7 planes, 4 = 7 planes and, in wj2, a copy
// of the wJ plane in the BP1.0 layout (BP3.0 and BP1.0 factors live at the
// same Gauss points, so one pass serves both); MIN: also the per-element
// minimum |J|.
template <int qn, int kind, bool MIN>
__device__ __forceinline__ void geofacs_body(int64_t E, const double *__restrict__ nodes,
                                             const double *__restrict__ weights, const double *__restrict__ verts,
                                             double *__restrict__ geo, double *__restrict__ detJ_min,
                                             double *__restrict__ wj2) {
    using C = GeoCfg<qn>;
    constexpr int QP = C::QP, qq = C::qq, EPB = C::EPB, PER = C::PER;
    extern __shared__ double smem[];
    double *sx = smem, *sw = sx + pad2(qn);
    long long *fx = reinterpret_cast<long long *>(sw + pad2(qn)), *fw = fx + pad2(qn);  // nodes, weights in 62 bits
    double *buf = reinterpret_cast<double *>(fw + pad2(qn));
    for (int t = threadIdx.x; t < qn; t += blockDim.x) {
        const double w = __ldg(weights + t);
        sx[t] = __ldg(nodes + t);
        sw[t] = w;
        fx[t] = __double2ll_rn(sx[t] * 0x1p62);
        fw[t] = geo_fixed(w, (__double2hiint(w) >> 20) - 1022);
    }
    const int64_t e0 = (int64_t)blockIdx.x * EPB;
    const int64_t nel = (E - e0) < EPB ? (E - e0) : EPB;
    for (int t = threadIdx.x; t < EPB * 24; t += blockDim.x) {
        const int el = t / 24, p = t % 24;
        buf[el * PER + p] = (el < nel) ? __ldg(verts + (e0 + el) * 24 + p) : 0.0;
    }
    __syncthreads();

    const int el = threadIdx.x / qq, ab = threadIdx.x % qq;
    const int u = ab % qn, v = ab / qn;
    const bool valid = el < nel;
    const int64_t e = e0 + el;
    const double *vx = buf + el * PER;  // vertices [c][d]
    double *K = buf + el * PER + 24;    // 36 map coefficients
    double *Xr = K + 36;                // dx/dr at (s_u, t_v): [u][v][d]
    double *Xs = Xr + 3 * qq;           // dx/ds at (r_u, t_v)
    double *Xt = Xs + 3 * qq;           // dx/dt at (r_u, s_v)
    double *sdet = Xt + 3 * qq;         // per-thread minimum |J|
    int *scale = reinterpret_cast<int *>(sdet + qq);  // |X_dir| < 2^scale[dir]; [3..6]: the element is left to FP64; [7]: G is

    // tabulate the three column tables of X.  Along r the map's derivative is
    // dx/dr(s, t) = 1/8 [ A (1-s)(1-t) + B (1+s)(1-t) + C (1-s)(1+t) + D (1+s)(1+t) ]
    // with the r-edge vectors A = x1 - x0, B = x3 - x2, C = x5 - x4,
    // D = x7 - x6, i.e. the bilinear form K0 + s K1 + t (K2 + s K3); the same
    // holds along s and t with their own edges.  The 3 x 4 x 3 coefficients
    // of an element are formed once (in shared memory), then each table entry
    // costs three FMAs per component.
    for (int ci = ab; ci < 36; ci += qq) {
        // K[(dir*4 + w)*3 + d]: dir 0 = r, 1 = s, 2 = t; w = coefficient
        const int dir = ci / 12, w = (ci / 3) % 4, d = ci % 3;
        // corner pairs (lower, upper) of the four edges along dir, in the
        // order (-,-), (+,-), (-,+), (+,+) of the two other coordinates
        const int stride = 1 << dir;
        int base[4];
        {
            const int o1 = (dir == 0) ? 2 : 1, o2 = (dir == 2) ? 2 : 4;
            base[0] = 0;
            base[1] = o1;
            base[2] = o2;
            base[3] = o1 + o2;
        }
        double ed[4];
#pragma unroll
        for (int h = 0; h < 4; h++) ed[h] = vx[(base[h] + stride) * 3 + d] - vx[base[h] * 3 + d];
        // (1-p)(1-q) A + (1+p)(1-q) B + (1-p)(1+q) C + (1+p)(1+q) D
        //   = (A+B+C+D) + p (B-A+D-C) + q (C+D-A-B) + p q (A-B-C+D)
        double kv;
        if (w == 0) kv = ed[0] + ed[1] + ed[2] + ed[3];
        else if (w == 1) kv = (ed[1] - ed[0]) + (ed[3] - ed[2]);
        else if (w == 2) kv = (ed[2] + ed[3]) - (ed[0] + ed[1]);
        else kv = (ed[0] - ed[1]) - (ed[2] - ed[3]);
        K[ci] = 0.125 * kv;
    }
    __syncthreads();
    // scales: a column's entries are bounded by the sum of its coefficients,
    // taken on their leading 21 bits, rounded up (three threads of an element
    // would keep the FP64 pipe as busy as all of them: 5 % of the FP64 path)
    for (int d = ab; d < 3; d += qq) {
        int most = 0, e3[3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            int hi[4], top = 0;
            bool any[4];
#pragma unroll
            for (int w = 0; w < 4; w++) {
                const double k = K[d * 12 + w * 3 + c];
                hi[w] = fx_abs_hi(k);
                any[w] = (hi[w] | __double2loint(k)) != 0;
                top = max(top, hi[w] >> 20);
            }
            int sum = 0;
#pragma unroll
            for (int w = 0; w < 4; w++)
                if (any[w]) sum += (((hi[w] & 0xfffff) | 0x100000) >> min(31, top - (hi[w] >> 20))) + 1;
            e3[c] = sum == 0 ? -10000 : fx_top(sum - 1) + top - 1043;
            most = c == 0 ? e3[0] : max(most, e3[c]);
        }
        bool left = false;
#pragma unroll
        for (int c = 0; c < 3; c++) left = left || (e3[c] != -10000 && e3[c] < most - kGeoRange);
        scale[d] = most;
        if (d == 0) scale[3] = scale[7] = 0;
        scale[4 + d] = left || most > 150 || most < -150;
    }
    __syncthreads();
    const int kr = scale[0], ks = scale[1], kt = scale[2];
    bool left = scale[4] | scale[5] | scale[6];
    long long *Fr = reinterpret_cast<long long *>(Xr), *Fs = reinterpret_cast<long long *>(Xs),
              *Ft = reinterpret_cast<long long *>(Xt);
    if (!left) {
        // at the element's centre, in binary32 and before any point is computed:
        // a left-handed element, or one with nearly parallel columns
        if (ab < 3) {
            const int d1 = ab == 2 ? 0 : ab + 1, d2 = ab == 0 ? 2 : ab - 1;
            float x[3], y[3], z[3];
#pragma unroll
            for (int c = 0; c < 3; c++) {
                x[c] = geo_float(K[ab * 12 + c], scale[ab]);
                y[c] = geo_float(K[d1 * 12 + c], scale[d1]);
                z[c] = geo_float(K[d2 * 12 + c], scale[d2]);
            }
            const float c0 = y[1] * z[2] - y[2] * z[1], c1 = y[2] * z[0] - y[0] * z[2], c2 = y[0] * z[1] - y[1] * z[0];
            if (c0 * c0 + c1 * c1 + c2 * c2 < 0x1p-7f || x[0] * c0 + x[1] * c1 + x[2] * c2 < 0x1p-7f) scale[3] = 1;
        }
        // entry (u, v): X_r at (s_u, t_v), X_s at (r_u, t_v), X_t at (r_u, s_v)
        const long long p = fx[u], w2 = fx[v];
#pragma unroll
        for (int dir = 0; dir < 3; dir++) {
            const int k = dir == 0 ? kr : dir == 1 ? ks : kt;
            long long *F = dir == 0 ? Fr : dir == 1 ? Fs : Ft;
#pragma unroll
            for (int d = 0; d < 3; d++) {
                const double *kk = K + dir * 12 + d;
                F[ab * 3 + d] = geo_fixed(kk[0], k) + geo_mul<2>(p, geo_fixed(kk[3], k)) +
                                geo_mul<2>(w2, geo_fixed(kk[6], k) + geo_mul<2>(p, geo_fixed(kk[9], k)));
            }
        }
    }
    __syncthreads();
    left = left || scale[3];

    // thread (a, b) = (u, v) walks the c direction
    const int a = u, b = v;
    const double wab = sw[a] * sw[b];
    double mindet = 1e300;
    double *ge = geo + (valid ? e : 0) * (kind == 1 ? 1 : 7) * (int64_t)QP + ab;
    if (valid && !left) {
        long long xt[3];
#pragma unroll
        for (int d = 0; d < 3; d++) xt[d] = Ft[(a + qn * b) * 3 + d];  // dx/dt at (r_a, s_b)
        // the weights' product, its leading bit at 61
        long long w2 = geo_mul<2>(fw[a], fw[b]);
        int kw = (__double2hiint(sw[a]) >> 20) + (__double2hiint(sw[b]) >> 20) - 2 * 1022;
        const int lead = __clzll(w2) - 2;
        w2 <<= lead;
        kw -= lead;
        const int K3 = kr + ks + kt;
        int least = 0x7fffffff;  // determinant's high word (negative: inverted)
        int most = 0, thin = 0x7fffffff;  // of the squares' high words: at 2^30 and above (long cofactors) they do not fit
#pragma unroll 1
        for (int c = 0; c < qn; c++) {
            long long xr[3], xs[3];
#pragma unroll
            for (int d = 0; d < 3; d++) {
                xr[d] = Fr[(b + qn * c) * 3 + d];  // dx/dr at (s_b, t_c)
                xs[d] = Fs[(a + qn * c) * 3 + d];  // dx/ds at (r_a, t_c)
            }
            // twice C_r = X_s x X_t
            long long cr[3] = {geo_cross(xs[1], xt[2], xs[2], xt[1]) << 1, geo_cross(xs[2], xt[0], xs[0], xt[2]) << 1,
                               geo_cross(xs[0], xt[1], xs[1], xt[0]) << 1};
            const long long det = geo_dot<0>(xr, cr);  // |J| = det 2^(K3 - 59)
            least = min(least, (int)(det >> 32));
            const int z = max(0, __clzll(det | 1) - 2);
            const long long W = geo_mul<2>(w2, fw[c]);  // weights 2^(62 - kwc)
            const int kwc = kw + (__double2hiint(sw[c]) >> 20) - 1022;
            const long long dn = det << z;
            const double wj = fx_to_double(geo_mul<2>(W, dn), kwc + K3 - 59 - z);
            if (MIN) mindet = fmin(mindet, fx_to_double(det, K3 - 59));
            if (kind == 1) {
                ge[c * qq] = wj;
            } else {
                long long cs[3] = {geo_cross(xt[1], xr[2], xt[2], xr[1]) << 1, geo_cross(xt[2], xr[0], xt[0], xr[2]) << 1,
                                   geo_cross(xt[0], xr[1], xt[1], xr[0]) << 1};
                long long ct[3] = {geo_cross(xr[1], xs[2], xr[2], xs[1]) << 1, geo_cross(xr[2], xs[0], xr[0], xs[2]) << 1,
                                   geo_cross(xr[0], xs[1], xr[1], xs[0]) << 1};
                const long long f = geo_mul<3>(W, geo_recip(dn));  // W / |J| = f 2^(kwc - 64 - K3 + z)
                const long long grr = geo_dot<2>(cr, cr), gss = geo_dot<2>(cs, cs), gtt = geo_dot<2>(ct, ct);
                most |= (int)(grr >> 32) | (int)(gss >> 32) | (int)(gtt >> 32);
                thin = min(thin, __vimin3_s32((int)(grr >> 32), (int)(gss >> 32), (int)(gtt >> 32)));
                // G = (f g / 2^61) 2^(kwc - K3 + z + E_a + E_b + 59), E_r = ks + kt - 61, ...
                const int k = kwc - K3 + z - 63;
                double *g = ge + c * qq;
                g[0 * QP] = fx_to_double(geo_mul<3>(f, grr), k + 2 * (ks + kt));
                g[1 * QP] = fx_to_double(geo_mul<3>(f, geo_dot<2>(cr, cs)), k + K3 + kt);
                g[2 * QP] = fx_to_double(geo_mul<3>(f, geo_dot<2>(cr, ct)), k + K3 + ks);
                g[3 * QP] = fx_to_double(geo_mul<3>(f, gss), k + 2 * (kr + kt));
                g[4 * QP] = fx_to_double(geo_mul<3>(f, geo_dot<2>(cs, ct)), k + K3 + kr);
                g[5 * QP] = fx_to_double(geo_mul<3>(f, gtt), k + 2 * (kr + ks));
                g[6 * QP] = wj;
                if (kind == 4) wj2[e * (int64_t)QP + c * qq + ab] = wj;
            }
        }
        if (least < 1 << (kGeoDet - 32)) scale[4] = 1;
        if (most >= 1 << 30 || most < 0 || thin < 1 << (kGeoSquare - 32)) scale[7] = 1;
    }
    __syncthreads();
    const bool all = scale[3] | scale[4] | scale[5] | scale[6];
    left = valid && (all || (kind != 1 && scale[7]));
    if (__syncthreads_or(left)) {
        // the same in FP64, for the elements that are left
        if (left) {
            // entry (u, v): X_r at (s_u, t_v), X_s at (r_u, t_v), X_t at (r_u, s_v)
            const double p = sx[u], w2 = sx[v];
#pragma unroll
            for (int d = 0; d < 3; d++) {
                Xr[ab * 3 + d] = fma(w2, fma(p, K[(0 * 4 + 3) * 3 + d], K[(0 * 4 + 2) * 3 + d]),
                                     fma(p, K[(0 * 4 + 1) * 3 + d], K[(0 * 4 + 0) * 3 + d]));
                Xs[ab * 3 + d] = fma(w2, fma(p, K[(1 * 4 + 3) * 3 + d], K[(1 * 4 + 2) * 3 + d]),
                                     fma(p, K[(1 * 4 + 1) * 3 + d], K[(1 * 4 + 0) * 3 + d]));
                Xt[ab * 3 + d] = fma(w2, fma(p, K[(2 * 4 + 3) * 3 + d], K[(2 * 4 + 2) * 3 + d]),
                                     fma(p, K[(2 * 4 + 1) * 3 + d], K[(2 * 4 + 0) * 3 + d]));
            }
        }
        __syncthreads();
        if (left) {
            if (all) mindet = 1e300;
            double xt[3];
#pragma unroll
            for (int d = 0; d < 3; d++) xt[d] = Xt[(a + qn * b) * 3 + d];  // dx/dt at (r_a, s_b)
#pragma unroll 1
            for (int c = 0; c < qn; c++) {
                double xr[3], xs[3];
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    xr[d] = Xr[(b + qn * c) * 3 + d];  // dx/dr at (s_b, t_c)
                    xs[d] = Xs[(a + qn * c) * 3 + d];  // dx/ds at (r_a, t_c)
                }
                // C_r = X_s x X_t
                const double Cr0 = xs[1] * xt[2] - xs[2] * xt[1];
                const double Cr1 = xs[2] * xt[0] - xs[0] * xt[2];
                const double Cr2 = xs[0] * xt[1] - xs[1] * xt[0];
                const double det = xr[0] * Cr0 + xr[1] * Cr1 + xr[2] * Cr2;
                const double W = wab * sw[c];
                if (MIN && all) mindet = fmin(mindet, det);
                if (kind == 1) {
                    ge[c * qq] = W * det;
                } else {
                    const double Cs0 = xt[1] * xr[2] - xt[2] * xr[1];
                    const double Cs1 = xt[2] * xr[0] - xt[0] * xr[2];
                    const double Cs2 = xt[0] * xr[1] - xt[1] * xr[0];
                    const double Ct0 = xr[1] * xs[2] - xr[2] * xs[1];
                    const double Ct1 = xr[2] * xs[0] - xr[0] * xs[2];
                    const double Ct2 = xr[0] * xs[1] - xr[1] * xs[0];
                    const double f = W * recip(det);
                    {
                        double *g = ge + c * qq;
                        g[0 * QP] = f * (Cr0 * Cr0 + Cr1 * Cr1 + Cr2 * Cr2);
                        g[1 * QP] = f * (Cr0 * Cs0 + Cr1 * Cs1 + Cr2 * Cs2);
                        g[2 * QP] = f * (Cr0 * Ct0 + Cr1 * Ct1 + Cr2 * Ct2);
                        g[3 * QP] = f * (Cs0 * Cs0 + Cs1 * Cs1 + Cs2 * Cs2);
                        g[4 * QP] = f * (Cs0 * Ct0 + Cs1 * Ct1 + Cs2 * Ct2);
                        g[5 * QP] = f * (Ct0 * Ct0 + Ct1 * Ct1 + Ct2 * Ct2);
                        if (all) {
                            g[6 * QP] = W * det;
                            if (kind == 4) wj2[e * (int64_t)QP + c * qq + ab] = W * det;
                        }
                    }
                }
            }
        }
    }
    if (MIN) {
        sdet[ab] = mindet;
        __syncthreads();
        for (int s = 1; s < qq; s *= 2) {
            if ((ab % (2 * s)) == 0 && ab + s < qq) sdet[ab] = fmin(sdet[ab], sdet[ab + s]);
            __syncthreads();
        }
        if (ab == 0 && valid) detJ_min[e] = sdet[0];
    }
}

// Resident blocks per SM that the register allocation must allow (64 and 80
// registers; at 17 points 1068 us with three, 1195 with five).
constexpr int geo_min_blocks(int qn) { return qn <= 10 ? 4 : 3; }

template <int qn, int kind, bool MIN>
__global__ void __launch_bounds__(GeoCfg<qn>::threads, geo_min_blocks(qn))
geofacs_kernel(int64_t E, const double *__restrict__ nodes, const double *__restrict__ weights,
               const double *__restrict__ verts, double *__restrict__ geo, double *__restrict__ detJ_min,
               double *__restrict__ wj2) {
    geofacs_body<qn, kind, MIN>(E, nodes, weights, verts, geo, detJ_min, wj2);
}

template <int qn, int kind, bool MIN>
constexpr auto geo_fn() {
    return &geofacs_kernel<qn, kind, MIN>;
}

template <int N>
struct GeoLaunch {
    static cudaError_t run(const fem_basis *b, int kind, int64_t E, const double *verts, double *geo,
                           double *detJ_min, cudaStream_t s) {
        const OpsLayout L{N + 1, N + 2};
        if (kind == FEM_GEO_BP35) {
            using C = GeoCfg<N + 1>;
            const int64_t blocks = (E + C::EPB - 1) / C::EPB;
            auto k = detJ_min ? geo_fn<N + 1, 2, true>() : geo_fn<N + 1, 2, false>();
            k<<<(unsigned)blocks, C::threads, C::smem, s>>>(E, b->d_ops + L.offR(), b->d_ops + L.offW(), verts,
                                                            geo, detJ_min, nullptr);
        } else {
            using C = GeoCfg<N + 2>;
            const int64_t blocks = (E + C::EPB - 1) / C::EPB;
            const double *x = b->d_ops + L.offRt(), *w = b->d_ops + L.offWt();
            auto k = (kind == FEM_GEO_BP1) ? (detJ_min ? geo_fn<N + 2, 1, true>() : geo_fn<N + 2, 1, false>())
                                           : (detJ_min ? geo_fn<N + 2, 3, true>() : geo_fn<N + 2, 3, false>());
            k<<<(unsigned)blocks, C::threads, C::smem, s>>>(E, x, w, verts, geo, detJ_min, nullptr);
        }
        return cudaGetLastError();
    }
};

template <int N>
struct GeoPairLaunch {
    static cudaError_t run(const fem_basis *b, int64_t E, const double *verts, double *G30, double *wJ,
                           cudaStream_t s) {
        const OpsLayout L{N + 1, N + 2};
        using C = GeoCfg<N + 2>;
        const int64_t blocks = (E + C::EPB - 1) / C::EPB;
        geo_fn<N + 2, 4, false>()<<<(unsigned)blocks, C::threads, C::smem, s>>>(
            E, b->d_ops + L.offRt(), b->d_ops + L.offWt(), verts, G30, nullptr, wJ);
        return cudaGetLastError();
    }
};

template <int N>
struct GeoPrepare {
    template <int qn, int kind, bool MIN>
    static cudaError_t one() {
        return cudaFuncSetAttribute(geo_fn<qn, kind, MIN>(), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    GeoCfg<qn>::smem);
    }
    static cudaError_t run() {
        cudaError_t e = cudaSuccess;
        if (e == cudaSuccess) e = one<N + 1, 2, false>();
        if (e == cudaSuccess) e = one<N + 1, 2, true>();
        if (e == cudaSuccess) e = one<N + 2, 1, false>();
        if (e == cudaSuccess) e = one<N + 2, 1, true>();
        if (e == cudaSuccess) e = one<N + 2, 3, false>();
        if (e == cudaSuccess) e = one<N + 2, 3, true>();
        if (e == cudaSuccess) e = one<N + 2, 4, false>();
        return e;
    }
};

}  // namespace

cudaError_t launch_geofacs(const fem_basis *b, int kind, int64_t E, const double *verts, double *geo,
                           double *detJ_min, cudaStream_t s) {
    return dispatch_degree<GeoLaunch>(b->host.N, b, kind, E, verts, geo, detJ_min, s);
}

cudaError_t launch_geofacs_gauss_pair(const fem_basis *b, int64_t E, const double *verts, double *G30, double *wJ,
                                      cudaStream_t s) {
    return dispatch_degree<GeoPairLaunch>(b->host.N, b, E, verts, G30, wJ, s);
}

cudaError_t prepare_geofacs(int N) { return dispatch_degree<GeoPrepare>(N); }

}  // namespace fem
