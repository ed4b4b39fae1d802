// FP64-accurate pair functions in 64-bit fixed point, for GB300's integer pipes.
//
// GB300 runs FP64 at 1/64 of the FP32 rate (a warp instruction occupies an SM's
// FP64 pipe for about 19 cycles), so an FP64 pair sum is bound by that pipe.  The
// integer multiply-add (32 x 32 + 64 bits) runs at half the FP32 rate, and a sum
// of pair terms needs absolute rather than relative accuracy: with the charges
// scaled by their largest and the lengths by a power of two, every quantity of
// the sum fits a 64-bit integer with at least FP64's resolution.
//
// Scaled lengths: r' = r / 2^e with r_cut' in (4, 8].  Coordinates are integers of
// unit 2^-59, modulo 2^64 (differences are exact), s = r'^2 has unit 2^-54.
//
// F(s) = erfc(a sqrt s) / sqrt s and G(s) = -2 dF/ds are completely monotone:
// around the right end of an interval every Taylor coefficient in
// y = (right - s) / width is positive, so their polynomials evaluate in unsigned
// arithmetic.  Each octave of s (1/8 to 64) is cut into 64 pieces; the piece and y
// come from the bits of s.  A piece keeps a degree-6 polynomial of F and a
// degree-7 polynomial of G through Chebyshev nodes; the leading coefficients are
// 64-bit, the last three 32-bit.  The Gaussian-charge correction
// erfc(r / gamma) / r = F_1(t) / gamma, t = s / gamma'^2, uses a second table of
// the same shape at a = 1.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace qeq {

using u32 = uint32_t;
using u64 = uint64_t;
using s32 = int32_t;
using s64 = int64_t;

#ifdef __CUDA_ARCH__
#define QEQ_FX __device__ __forceinline__
#else
#define QEQ_FX __host__ __device__ __forceinline__
#endif

constexpr int kFxCoordBits = 59;   // unit of scaled coordinates: 2^-59
constexpr int kFxSigmaBits = 56;   // unit of scaled sigma^2: 2^-56
constexpr u64 kFxSigmaSat = 1ull << 61;  // sigma'^2 of 32 or more: the exact path
constexpr int kFxSub = 64;         // pieces per octave
constexpr int kFxLzTop = 4;        // leading zeros of the high word of s in [32, 64)
constexpr int kFxLzMin = 12;       // ... in [1/8, 1/4), the lowest octave of the pair table
constexpr int kFxLzMinCorr = 11;   // ... in [1/4, 1/2), the lowest of the correction table
constexpr int kFxOctaves = kFxLzMin - kFxLzTop + 1;
constexpr int kFxRowWords = 7;     // 16-byte words of a piece
constexpr int kFxFBits = 59;       // unit of F (both tables): 2^-59
constexpr int kFxGBits = 60;       // unit of G 2^-b, b = fx_bshift(lz) (pair table), and of G_1
// The 32-bit coefficients have coarser units: F's by 2^3, G's by 2^1 (pair table)
// and 2^3 (correction table).
constexpr int kFxFShift = 3, kFxGShift = 1, kFxG1Shift = 3;
// Corrections beyond t = 36, r / gamma = 6 (below 2e-17 / r) are dropped, so the
// correction table keeps seven octaves from 1/4 and the first pieces of [32, 64).
constexpr int kFxCorrRows = 7 * kFxSub + 16;

// G reaches 22.6 at s = 1/8, where the differences are below 1/2: in the three lowest
// octaves (s < 1) the table holds G 2^-b and the differences are shifted by b.
QEQ_FX int fx_bshift(int lz) { return lz < 10 ? 0 : lz == 10 ? 1 : lz == 11 ? 2 : 4; }

// Words and 32 x 32 + 64 bit products by name: as 64-bit expressions the compiler
// merges a word's extraction with its extension and multiplies 64 by 64 bits
// (twice the instructions).
#ifdef __CUDA_ARCH__
QEQ_FX u32 fx_hi(u64 a) {
    u32 l, h;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "l"(a));
    return h;
}
QEQ_FX u32 fx_lo(u64 a) {
    u32 l, h;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(l), "=r"(h) : "l"(a));
    return l;
}
QEQ_FX u64 fx_wide(u32 a, u32 b, u64 c) {
    u64 r;
    asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
QEQ_FX s64 fx_wide(s32 a, s32 b, s64 c) {
    s64 r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
#else
QEQ_FX u32 fx_hi(u64 a) { return (u32)(a >> 32); }
QEQ_FX u32 fx_lo(u64 a) { return (u32)a; }
QEQ_FX u64 fx_wide(u32 a, u32 b, u64 c) { return (u64)a * b + c; }
QEQ_FX s64 fx_wide(s32 a, s32 b, s64 c) { return (s64)((u64)((s64)a * b) + (u64)c); }
#endif
QEQ_FX s32 fx_his(s64 a) { return (s32)fx_hi((u64)a); }
QEQ_FX int fx_clz(u32 a) {
#ifdef __CUDA_ARCH__
    return __clz((int)a);
#else
    return a ? __builtin_clz(a) : 32;
#endif
}
// high word of a b, plus c
QEQ_FX u32 fx_mulhi_add(u32 a, u32 b, u32 c) {
#ifdef __CUDA_ARCH__
    u32 r;
    asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
#else
    return (u32)(((u64)a * b) >> 32) + c;
#endif
}
// (a b) >> 64 of unsigned operands, at most 2 units low
QEQ_FX u64 fx_mulhi(u64 a, u64 b) {
    const u32 m0 = fx_mulhi_add(fx_hi(a), fx_lo(b), 0u), m1 = fx_mulhi_add(fx_lo(a), fx_hi(b), 0u);
    return fx_wide(fx_hi(a), fx_hi(b), (u64)m0 + m1);
}

// One Horner step c + y p, y = (X + XL 2^-32) 2^-32, a few units of truncation low.
// Explicit carry chains: 64-bit additions of zero-extended words would cost moves.
QEQ_FX u64 fx_step(u64 c, u32 X, u32 XL, u64 p) {
#ifdef __CUDA_ARCH__
    u64 r;
    asm("{\n\t"
        ".reg .u32 pl, ph, cl, chh, t, r0, r1;\n\t"
        "mov.b64 {pl, ph}, %4;\n\t"
        "mov.b64 {cl, chh}, %1;\n\t"
        "mul.hi.u32 t, %2, pl;\n\t"
        "mad.hi.cc.u32 r0, %3, ph, cl;\n\t"
        "addc.u32 r1, chh, 0;\n\t"
        "add.cc.u32 r0, r0, t;\n\t"
        "addc.u32 r1, r1, 0;\n\t"
        "mad.lo.cc.u32 r0, %2, ph, r0;\n\t"
        "madc.hi.u32 r1, %2, ph, r1;\n\t"
        "mov.b64 %0, {r0, r1};\n\t"
        "}"
        : "=l"(r)
        : "l"(c), "r"(X), "r"(XL), "l"(p));
    return r;
#else
    const u32 th = fx_hi((u64)X * fx_lo(p));
    const u32 tl = fx_mulhi_add(XL, fx_hi(p), 0u);
    const u64 r = c + th + tl;
    return r + (u64)X * fx_hi(p);
#endif
}

// A piece: six 16-byte words of coefficients (16-byte loads) and one of padding, so
// that the rows of a table start in all eight 16-byte columns of the shared-memory
// banks (six words, 96 bytes, would use only every other one).
struct alignas(16) FxRow {
    u64 f0, f1, f2, f3;
    u32 f4, f5, f6, g5;
    u64 g0, g1, g2, g3, g4;
    u32 g6, g7;
    u64 pad[2];
};
static_assert(sizeof(FxRow) == 16 * kFxRowWords, "a piece is seven 16-byte words");

template <bool WITH_G, int GSHIFT>
QEQ_FX void fx_eval(const FxRow &c, u32 X, u32 XL, u64 &F, u64 &G) {
    const u32 q4 = fx_mulhi_add(X, fx_mulhi_add(X, c.f6, c.f5), c.f4);
    u64 p = c.f3 + (fx_wide(X, q4, 0ull) >> (32 - kFxFShift));
    p = fx_step(c.f2, X, XL, p);
    p = fx_step(c.f1, X, XL, p);
    F = fx_step(c.f0, X, XL, p);
    if (WITH_G) {
        const u32 q5 = fx_mulhi_add(X, fx_mulhi_add(X, c.g7, c.g6), c.g5);
        p = c.g4 + (fx_wide(X, q5, 0ull) >> (32 - GSHIFT));
        p = fx_step(c.g3, X, XL, p);
        p = fx_step(c.g2, X, XL, p);
        p = fx_step(c.g1, X, XL, p);
        G = fx_step(c.g0, X, XL, p);
    }
}

// Piece and position of s (high word hi, leading zeros lz): y = ~(bits below the piece's).
QEQ_FX int fx_piece(u32 hi, int lz) { return (int)(hi >> (25 - lz)) + (kFxLzMin - 1 - lz) * kFxSub; }
QEQ_FX u64 fx_pos(u64 s, int lz) { return ~(s << (lz + 7)); }

// 1 / gamma' and 1 / gamma'^2 of gamma'^2 = g2 2^-56 (0 < g2 < 2^62): with
// z = clz(g2) rounded down to even, 1 / gamma' = IG 2^(z/2 - 66) and
// 1 / gamma'^2 = IG2 2^(z - 68).  A 24-bit reciprocal square root M 2^-39 of the
// leading bits, its residual e = 1 - M^2 gn 2^-110 exactly (modulo 2^64, in units
// of 2^-78), and the series M (1 + e / 2 + 3 e^2 / 8): relative error below 2^-51.
QEQ_FX void fx_inv_gamma(u64 g2, int &z, u64 &IG, u64 &IG2) {
    const u32 h = fx_hi(g2);
    z = (h ? fx_clz(h) : 32 + fx_clz(fx_lo(g2))) & ~1;
    const u64 gn = g2 << z;
#ifdef __CUDA_ARCH__
    const float gf = (float)fx_hi(gn);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(gf));
    const u32 M = __float2uint_rn(y * 0x1p39f);
#else
    const u32 M = (u32)(0x1p39 / __builtin_sqrt((double)fx_hi(gn)) + 0.5);
#endif
    const u64 m2 = fx_wide(M, M, 0ull);
    u64 w = fx_wide(fx_hi(gn), fx_lo(m2), (u64)fx_mulhi_add(fx_lo(gn), fx_lo(m2), 0u));
    w = fx_wide(fx_lo(gn), fx_hi(m2), w);
    w += (u64)(fx_hi(gn) * fx_hi(m2)) << 32;
    const s64 e = -(s64)w;             // unit 2^-78, below 2^57
    const s32 e1 = (s32)(e >> 26);     // unit 2^-52
    const s32 e2 = e1 >> 16;           // unit 2^-36
    IG = ((u64)M << 39) + (u64)(fx_wide((s32)M, e1, 0ll) >> 14) + (fx_wide(M, (u32)(3 * e2 * e2), 0ull) >> 36);
    IG2 = fx_mulhi(IG, IG);
}

// A double as an integer of unit 2^-bits, modulo 2^64 (bits below the unit are
// rounded off; infinities and NaNs give 0).
QEQ_FX u64 fx_from_double(double x, int bits) {
    u64 b;
#ifdef __CUDA_ARCH__
    b = (u64)__double_as_longlong(x);
#else
    __builtin_memcpy(&b, &x, sizeof b);
#endif
    const int ex = (int)(b >> 52) & 0x7FF;
    const u64 m = (b & 0xFFFFFFFFFFFFFull) | ((u64)(ex != 0) << 52);
    const int sh = (ex ? ex : 1) - 1075 + bits;
    u64 r = 0;
    if (ex == 0x7FF)
        r = 0;
    else if (sh >= 0)
        r = sh < 64 ? m << sh : 0ull;
    else if (sh > -55)
        r = (m + (1ull << (-sh - 1))) >> -sh;
    return b >> 63 ? 0ull - r : r;
}

// sigma^2 of unit 2^-56 in scaled lengths (bits = 56 - 2 e), saturated; a NaN
// sigma takes no correction.
QEQ_FX u64 fx_sigma2(double sigma, int bits) {
    const double s2 = sigma * sigma;
    if (!(s2 == s2)) return 0ull;
    const double cap = 32.0;  // sigma'^2
#ifdef __CUDA_ARCH__
    const double lim = __hiloint2double((1023 + kFxSigmaBits - bits) << 20, 0) * cap;
#else
    const double lim = __builtin_ldexp(cap, kFxSigmaBits - bits);
#endif
    if (!(s2 < lim)) return kFxSigmaSat;
    return fx_from_double(s2, bits);
}

// Signed numbers below 2^62 are multiplied by their high words (30 bits and sign) and
// their low words less the last two bits (fx_low), with value
// h 2^32 + l 2^2: a b = ah bh 2^64 + (ah bl + al bh) 2^34, each 32 x 32 product one
// multiply-add into a 64-bit sum.  The low words' product, between 0 and 1 unit of the
// high words' (which typical terms, far below full scale, would notice), enters by
// its high word.
constexpr int kFxCross = 30;  // the cross sum's unit is 2^-30 of the high sum's
QEQ_FX s32 fx_low(u64 a) { return (s32)(fx_lo(a) >> 2); }

// q as an integer of unit 2^(Eq - qbits), Eq = e0 - 1022 with e0 the largest biased
// exponent of the charges: |q| < 2^Eq, so |result| < 2^qbits.
QEQ_FX s64 fx_charge(double q, int e0, int qbits) { return (s64)fx_from_double(q, 1022 - e0 + qbits); }

// Squared distance of unit 2^-54 from differences of unit 2^-59 (modulo 2^64 when
// the distance exceeds 32).
QEQ_FX u64 fx_dist2(s64 dx, s64 dy, s64 dz) {
    const s32 hx = fx_his(dx), hy = fx_his(dy), hz = fx_his(dz);
    const s32 lx = fx_low((u64)dx), ly = fx_low((u64)dy), lz = fx_low((u64)dz);
    const s64 sq = fx_wide(hx, hx, fx_wide(hy, hy, fx_wide(hz, hz, 1ll)));
    const s64 cr = fx_wide(hx, lx, fx_wide(hy, ly, fx_wide(hz, lz, 1ll << (kFxCross - 2))));
    return (u64)sq + (u64)(cr >> (kFxCross - 1));
}

// Gaussian-charge correction of a pair at s with gamma'^2 = g2: F and G 2^-b lose
// it (b = fx_bshift of s).  False where its table does not reach (t < 1/4).
template <bool WITH_G>
QEQ_FX bool fx_correct(const FxRow *corr, u64 s, int b, u64 g2, s64 &F, s64 &G) {
    int z;
    u64 IG, IG2;
    fx_inv_gamma(g2, z, IG, IG2);
    // t = s / gamma'^2 of unit 2^-54: (s 2^(z-4)) IG2 2^-64
    const u64 t = fx_mulhi(z >= 4 ? s << (z - 4) : s >> (4 - z), IG2);
    const u32 th = fx_hi(t);
    const int lz = fx_clz(th);
    if (lz > kFxLzMinCorr || lz < kFxLzTop) return lz < kFxLzTop;
    const u64 y = fx_pos(t, lz);
    u64 f1, g1 = 0;
    int row = fx_piece(th, lz) - (kFxLzMin - kFxLzMinCorr) * kFxSub;
    row = row < kFxCorrRows - 1 ? row : kFxCorrRows - 1;
    fx_eval<WITH_G, kFxG1Shift>(corr[row], fx_hi(y), fx_lo(y), f1, g1);
    // f1 / gamma' of unit 2^-59, g1 / gamma'^3 2^-b of unit 2^-60 (g1 normalised first)
    const int shf = z / 2 - 2;
    const u64 fc = fx_mulhi(f1, IG);
    F -= (s64)(shf >= 0 ? fc << shf : fc >> -shf);
    if (WITH_G) {
        const int k = fx_clz(fx_hi(g1) | 1u);
        const u64 gc = fx_mulhi(fx_mulhi(g1 << k, IG), IG2);
        const int sh = k + b + 6 - 3 * (z / 2);
        G -= (s64)(sh >= 0 ? (sh < 64 ? gc >> sh : 0ull) : gc << -sh);
    }
    return true;
}

// A sum of products: high words' and cross products.  The cross sum takes four
// products (each below 2^61 - a field term's |d'| g' stays below that: g' is half its
// range where d' may be full) before fold() moves its whole units into the high sum;
// its remainder stays, so nothing is lost.
struct FxSum {
    s64 h = 0, m = 0;
    // b's low word as fx_low
    QEQ_FX void add(u64 a, s32 bh, s32 bl) {
        h = fx_wide(fx_his((s64)a), bh, h);
        m = fx_wide(fx_his((s64)a), bl, fx_wide(fx_low(a), bh, m));
        m += (s64)(u64)fx_mulhi_add(fx_lo(a), (u32)bl, 0u);
    }
    QEQ_FX void fold() {
        h += m >> kFxCross;
        m &= (1ll << kFxCross) - 1;
    }
};

// (a b) >> (64 - up), b's low word as fx_low.
QEQ_FX s64 fx_mul(u64 a, s32 bh, s32 bl, int up) {
    const u32 ll = fx_mulhi_add(fx_lo(a), (u32)bl, 1u << (kFxCross - up - 1));
    const s64 m = fx_wide(fx_his((s64)a), bl, fx_wide(fx_low(a), bh, (s64)(u64)ll));
    return (fx_wide(fx_his((s64)a), bh, 0ll) << up) + (m >> (kFxCross - up));
}

}  // namespace qeq
