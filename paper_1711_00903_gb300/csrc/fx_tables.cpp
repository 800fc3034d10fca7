// Host side of the fixed-point operators: see fx_layout.h and fx.cuh.
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <mutex>

#include "fx_layout.h"

namespace fem {
namespace {

int g_violations = 0;

// round(A 2^(64 - tau)) for |A| <= 2^tau: exact for entries above 2^(tau - 11).
__int128 scaled(double a, int tau) {
    int e;
    const double m = std::frexp(a, &e);
    const __int128 r = (__int128)std::llrint(std::ldexp(m, 53));
    const int sh = e - 53 + 64 - tau;
    if (sh >= 0) return r * ((__int128)1 << sh);
    if (sh < -100) return 0;
    return (r + ((__int128)1 << (-sh - 1))) >> -sh;
}

FxEntry halves(__int128 c, int *bad) {
    const __int128 h = (c + ((__int128)1 << 31)) >> 32;
    if (h > INT32_MAX || h < INT32_MIN) ++*bad;
    FxEntry e;
    e.h = (int)(int64_t)h;
    e.l = (int)(uint32_t)(uint64_t)c;
    return e;
}

// Folds A (P x Q, row-major, parity sig) scaled by 2^-tau into out; returns the number
// of bounds that do not hold.
int fold_scaled(int P, int Q, int sig, const double *A, int bits, double room, int tau, FxEntry *out) {
    int bad = 0;
    const int hp = P / 2, hq = Q / 2;
    // the entry with its image under the operator's symmetry: the mean of the
    // two is nearer to the exact entry than either
    auto I = [&](int a, int i) {
        const __int128 x = scaled(A[a * Q + i], tau), y = scaled(A[(P - 1 - a) * Q + (Q - 1 - i)], tau);
        return (x + (sig > 0 ? y : -y)) >> 1;
    };
    FxEntry *S = out, *T = out + hp * hq, *cm = T + hp * hq, *rm = cm + (Q % 2 ? hp : 0);
    // bounds of a row's sums, with |e| <= room 2^(bits + 1): the sum of the high
    // products and that of the cross products below 2^63
    auto check = [&](const FxEntry *r, int n, const FxEntry *extra) {
        double h = 0.0, l = 0.0;
        for (int i = 0; i < n; i++) {
            h += std::fabs((double)r[i].h);
            l += std::fabs((double)r[i].l);
        }
        if (extra) {
            h += std::fabs((double)extra->h);
            l += std::fabs((double)extra->l);
        }
        const double xh = room * std::ldexp(1.0, bits + 1 - 32), lim = std::ldexp(1.0, 63) - std::ldexp(1.0, 32);
        if (h * xh >= lim || h * std::ldexp(1.0, 31) + l * xh >= lim) bad++;
    };
    for (int a = 0; a < hp; a++)
        for (int i = 0; i < hq; i++) {
            S[a * hq + i] = halves((I(a, i) + I(a, Q - 1 - i))  >> 1, &bad);
            T[a * hq + i] = halves((I(a, i) - I(a, Q - 1 - i)) >> 1, &bad);
        }
    if (Q % 2)
        for (int a = 0; a < hp; a++) cm[a] = halves(I(a, hq) >> 1, &bad);
    if (P % 2) {
        for (int i = 0; i < hq; i++) rm[i] = halves(I(hp, i), &bad);
        if (Q % 2) rm[hq] = halves(I(hp, hq) >> 1, &bad);
        check(rm, hq, Q % 2 ? rm + hq : nullptr);
    }
    for (int a = 0; a < hp; a++) {
        check(S + a * hq, hq, Q % 2 ? cm + a : nullptr);
        check(T + a * hq, hq, nullptr);
    }
    return bad;
}

// At kAutoTau, the smallest tau whose scaled rows hold the bounds: a row's
// absolute sum at most 2^tau, up to 2 % over (the outputs have that room),
// every entry's high half within 32 bits.
constexpr int kAutoTau = -1;
int fold(int P, int Q, int sig, const double *A, int bits, double room, int tau, FxEntry *out) {
    if (tau != kAutoTau) {
        g_violations += fold_scaled(P, Q, sig, A, bits, room, tau, out);
        return tau;
    }
    double nu = 0.0;
    for (int a = 0; a < P; a++) {
        double s = 0.0;
        for (int i = 0; i < Q; i++) s += std::fabs(A[a * Q + i]);
        nu = s > nu ? s : nu;
    }
    std::frexp(nu / 1.02, &tau);
    int bad = fold_scaled(P, Q, sig, A, bits, room, tau, out);
    for (int up = 0; bad && up < 2; up++) bad = fold_scaled(P, Q, sig, A, bits, room, ++tau, out);
    g_violations += bad;
    return tau;
}

int exponent(double w) { return std::ilogb(w) + 1; }

}  // namespace

const FxTables &fx_tables() {
    static FxTables *t = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        t = new FxTables();
        for (int N = 1; N <= kMaxN; N++) {
            HostBasis hb;
            compute_basis(N, &hb);
            const int n = N + 1, m = N + 2;
            FxDegree &d = t->d[N];
            for (int i = 0; i < n; i++) d.wn[i] = exponent(hb.w[i < n - 1 - i ? i : n - 1 - i]);
            for (int i = 0; i < m; i++) d.wm[i] = exponent(hb.wt[i < m - 1 - i ? i : m - 1 - i]);
            double IT[kMaxQ * kMaxQ], DT[kMaxQ * kMaxQ], DtT[kMaxQ * kMaxQ];
            for (int a = 0; a < m; a++)
                for (int i = 0; i < n; i++) IT[i * m + a] = std::ldexp(hb.I[a * n + i], d.wm[a] - d.wn[i]);
            for (int a = 0; a < n; a++)
                for (int i = 0; i < n; i++) DT[i * n + a] = std::ldexp(hb.D[a * n + i], d.wn[a] - d.wn[i]);
            for (int a = 0; a < m; a++)
                for (int b = 0; b < m; b++) DtT[b * m + a] = std::ldexp(hb.Dt[a * m + b], d.wm[a] - d.wm[b]);
            const double *ops[kFoldCount] = {hb.I, IT, hb.D, DT, hb.Dt, DtT};
            for (int op = 0; op < kFoldCount; op++)
                d.tau[op] =
                    op == kFoldI
                        ? fold(m, n, 1, hb.I, fx_qbits30(N), N >= 7 ? 1.5 : 1.08, 1, t->c + fold_offset(N, op))
                        : fold(fold_rows(op, n, m), fold_cols(op, n, m), op == kFoldIT ? 1 : -1, ops[op],
                               op == kFoldD    ? fx_bits35(N) - 1
                               : op == kFoldDT ? fx_bits35(N)
                               : op == kFoldDt ? fx_qbits30(N)
                                               : kFxBits30,
                               op == kFoldDt   ? (N >= 7 ? 1.25 : 1.0)
                               : op == kFoldIT ? 1.08
                                               : 1.0,
                               kAutoTau, t->c + fold_offset(N, op));
        }
    });
    return *t;
}

int fx_table_violations() {
    fx_tables();
    return g_violations;
}

}  // namespace fem
