// Host side of fixed64.cuh: the piecewise tables in long double, rounded to the
// rows' integer units.
#pragma once

#include <cmath>
#include <vector>

#include "fixed64.cuh"

namespace qeq {

// Monomial coefficients in y of the polynomial of degree n - 1 that interpolates v
// at the n Chebyshev nodes y_k = (1 + cos(pi (k + 1/2) / n)) / 2: the Chebyshev
// series of the values, then the shifted polynomials T*_j(y) = T_j(2 y - 1), whose
// coefficients are integers (T*_{j+1} = (4 y - 2) T*_j - T*_{j-1}).
inline void fx_fit(int n, const long double *v, long double *c) {
    const long double pi = 3.141592653589793238462643383279502884L;
    long double prev[9] = {1.0L}, cur[9] = {-1.0L, 2.0L};  // T*_0, T*_1
    for (int m = 0; m < n; ++m) c[m] = 0.0L;
    for (int j = 0; j < n; ++j) {
        long double a = 0.0L;
        for (int k = 0; k < n; ++k) a += v[k] * cosl(pi * j * (k + 0.5L) / n);
        a *= (j == 0 ? 1.0L : 2.0L) / n;
        const long double *t = j == 0 ? prev : cur;
        for (int m = 0; m <= j; ++m) c[m] += a * t[m];
        if (j >= 1) {
            long double next[9] = {0.0L};
            for (int m = 0; m <= j; ++m) {
                if (m + 1 < 9) next[m + 1] += 4.0L * cur[m];
                next[m] -= 2.0L * cur[m];
            }
            for (int m = 0; m < 9; ++m) {
                next[m] -= prev[m];
                prev[m] = cur[m];
                cur[m] = next[m];
            }
        }
    }
}

inline u64 fx_round(long double c, int bits) {
    const long double x = ldexpl(c, bits) + 0.5L;
    return x > 0.0L ? (u64)x : 0ull;
}

// Table of F and G at screening a, piece order of fx_piece (lowest octave first),
// octaves up to [32, 64); gbits the unit of G, b_shift: G times 2^-b of its octave.
inline void fx_build(long double a, int lz_min, int gbits, bool b_shift, int gshift,
                     std::vector<FxRow> &out) {
    const long double pi = 3.141592653589793238462643383279502884L;
    constexpr int NF = 7, NG = 8;
    out.assign((size_t)kFxOctaves * kFxSub, FxRow{});
    for (int lz = kFxLzTop; lz <= lz_min; ++lz) {
        const long double lo = ldexpl(1.0L, 5 - (lz - kFxLzTop)), h = lo / kFxSub;
        for (int j = 0; j < kFxSub; ++j) {
            const long double right = lo + (j + 1) * h;
            long double vf[NF], vg[NG], cf[NF], cg[NG];
            auto eval = [&](long double y, long double &F, long double &G) {
                const long double s = right - y * h, r = sqrtl(s);
                F = erfcl(a * r) / r;
                G = (F + 2.0L * a / sqrtl(pi) * expl(-a * a * s)) / s;
                if (b_shift) G = ldexpl(G, -fx_bshift(lz));
            };
            long double F, G;
            for (int k = 0; k < NF; ++k) {
                eval(0.5L * (1.0L + cosl(pi * (k + 0.5L) / NF)), F, G);
                vf[k] = F;
            }
            for (int k = 0; k < NG; ++k) {
                eval(0.5L * (1.0L + cosl(pi * (k + 0.5L) / NG)), F, G);
                vg[k] = G;
            }
            fx_fit(NF, vf, cf);
            fx_fit(NG, vg, cg);
            FxRow r{};
            // the truncation of the evaluation is on average 4 units low in F, 3 in G
            r.f0 = fx_round(cf[0], kFxFBits) + 4;
            r.f1 = fx_round(cf[1], kFxFBits);
            r.f2 = fx_round(cf[2], kFxFBits);
            r.f3 = fx_round(cf[3], kFxFBits);
            r.f4 = (u32)fx_round(cf[4], kFxFBits - kFxFShift);
            r.f5 = (u32)fx_round(cf[5], kFxFBits - kFxFShift);
            r.f6 = (u32)fx_round(cf[6], kFxFBits - kFxFShift);
            r.g0 = fx_round(cg[0], gbits) + 3;
            r.g1 = fx_round(cg[1], gbits);
            r.g2 = fx_round(cg[2], gbits);
            r.g3 = fx_round(cg[3], gbits);
            r.g4 = fx_round(cg[4], gbits);
            r.g5 = (u32)fx_round(cg[5], gbits - gshift);
            r.g6 = (u32)fx_round(cg[6], gbits - gshift);
            r.g7 = (u32)fx_round(cg[7], gbits - gshift);
            out[(size_t)(kFxLzMin - lz) * kFxSub + j] = r;
        }
    }
}

// The pair table at the scaled screening a and the correction table.
inline void fx_build_tables(double a, std::vector<FxRow> &pair, std::vector<FxRow> &corr) {
    fx_build(a, kFxLzMin, kFxGBits, true, kFxGShift, pair);
    fx_build(1.0L, kFxLzMinCorr, kFxGBits, false, kFxG1Shift, corr);
    corr.erase(corr.begin(), corr.begin() + (kFxLzMin - kFxLzMinCorr) * kFxSub);
    corr.resize(kFxCorrRows);
}

// Exponent e of the scaled lengths r / 2^e for a cutoff: r_cut / 2^e in (4, 8].
inline int fx_exponent(double r_cut) {
    int e;
    const double m = std::frexp(r_cut, &e);  // r_cut = m 2^e, m in [0.5, 1)
    return m == 0.5 ? e - 4 : e - 3;
}

}  // namespace qeq
