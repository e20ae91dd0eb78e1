// Fixed-point arithmetic for the event loops of the likelihood kernels, at four
// to six integer instructions per product.
//
// A 64 x 64 -> high 64-bit signed product takes fourteen instructions (four
// 32 x 32 -> 64-bit products, their carries, the corrections for the signs).
// Here a value x is kept as Fx {h, l}, x = h 2^32 + l with both halves signed, and
//   a b 2^-64 ~ a.h b.h + hi32(a.h b.l) + hi32(b.h a.l) + 1,
// two 32-bit high products chained by their addends and one 32 x 32 -> 64-bit
// multiply-add.  Dropped: the product of the low halves (within 1/4 unit) and the
// fractions of the two high products, which the +1 centres: the error lies within
// 1.25 units of the result, 0.41 rms.  For Q62 operands a unit is 2^-60, 128
// times below the rounding of a double near 1.
//
// The functions are branch-free; outside their ranges (fx_angles_ok, fx_exp)
// their values are unspecified, every shift stays below 64 and every table
// index inside its table.
#pragma once

#include "int_math.cuh"
#include "ipa_internal.cuh"

namespace ipa {

struct Fx {
    int h, l;
};
// x < 2^63 - 2^31 (from there on h would be 2^31): a magnitude that fills 63 bits goes in negated.
__device__ __forceinline__ Fx fx(long long x) {
    return Fx{(int)(x >> 32) + (int)((unsigned)x >> 31), (int)x};
}

// acc + a b 2^-64 without the centring: exact for a zero operand, otherwise a unit
// low on average (sums of many products correct for their number).
__device__ __forceinline__ long long fx_mad0(Fx a, Fx b, long long acc) {
    const int m = __mulhi(a.h, b.l) + __mulhi(b.h, a.l);
    return ((long long)a.h * b.h + (long long)m) + acc;
}
// acc + a b 2^-64
__device__ __forceinline__ long long fx_mad(Fx a, Fx b, long long acc) {
    const int m = __mulhi(a.h, b.l) + (__mulhi(b.h, a.l) + 1);
    return ((long long)a.h * b.h + (long long)m) + acc;
}
// acc + a b 2^-64, `one` = (a != 0): centred, and exact for a = 0
__device__ __forceinline__ long long fx_mad1(Fx a, Fx b, long long acc, int one) {
    const int m = __mulhi(a.h, b.l) + (__mulhi(b.h, a.l) + one);
    return ((long long)a.h * b.h + (long long)m) + acc;
}
// a b for Q62 operands, in Q62
__device__ __forceinline__ long long fx_q62(Fx a, Fx b) {
    return (long long)((unsigned long long)fx_mad(a, b, 0) << 2);
}

// |x| 2^(63 - top) for a double's bits, |x| < 2^top (truncated; 0 where it underflows, and for 0).
__device__ __forceinline__ unsigned long long fx_magnitude(unsigned long long b, int top) {
    const unsigned long long M = ((b << 10) & 0x3FFFFFFFFFFFFFFFull) | 0x4000000000000000ull;   // 1.m in Q62
    const int s = top - 1 - ((int)((b >> 52) & 0x7FFull) - 1023);
    return M >> (s > 63 ? 63 : (s & 63));
}
__device__ __forceinline__ long long fx_signed(double x, int top) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const long long v = (long long)fx_magnitude(b, top);
    return (long long)b < 0 ? -v : v;
}

// x in fixed point with `top` (as above), rounded to an odd multiple of the last
// place (0 for 0): off by less than a unit either way, so that a sum of many has
// no bias, for one instruction more than truncation.
__device__ __forceinline__ long long fx_odd(double x, int top) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    unsigned long long m = fx_magnitude(b, top);
    m |= (unsigned long long)(m != 0ull);
    return (long long)b < 0 ? -(long long)m : (long long)m;
}

// v 2^(e2 - 62) as a double, rounded to nearest (halves away from zero; +0 for 0; the
// result must be normal).  Half of q62_to_double's instructions.
__device__ __forceinline__ double fx_to_double(long long v, int e2) {
    const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)a);
    const unsigned long long m = ((a << (lz & 63)) >> 11) + (((a << (lz & 63)) >> 10) & 1ull);
    const unsigned hi = (unsigned)(1023 + e2 - lz) << 20;                     // the hidden bit adds one
    const unsigned long long b = m + ((unsigned long long)(hi | (unsigned)((unsigned long long)v >> 32 & 0x80000000u)) << 32);
    return v == 0 ? 0.0 : __longlong_as_double((long long)b);
}

namespace fxc {
// sin and cos of (pi/32) f, |f| <= 1/2: Taylor coefficients (pi/32)^n / n!,
// rounded once, at the scale in the comment; terms past n = 9 are below 2^-70
constexpr long long kS1 = 0x6487ED5110B4611All;   // 2^66
constexpr long long kS3 = 0x295779CC4B7CA57Dll;   // 2^74
constexpr int kS5 = 1369108894;                   // 2^54
constexpr int kS7 = 80431924;                     // 2^62
constexpr int kS9 = 10767;                        // 2^62
constexpr long long kC2 = 0x4EF4F326F9177969ll;   // 2^70
constexpr long long kC4 = 0x40F07C206D6B0ECDll;   // 2^80
constexpr int kC6 = 358431870;                    // 2^58
constexpr int kC8 = 61691;                        // 2^58
// 2^(f/64) - 1, 0 <= f < 1: (ln2 / 64)^n / n!; terms past n = 6 are below 2^-58
constexpr long long kE1 = 0x58B90BFBE8E7BCD6ll;   // 2^69
constexpr long long kE2 = 0x3D7F7BFF058B1D51ll;   // 2^76
constexpr long long kE3 = 0x38D611AE09417F16ll;   // 2^84
constexpr int kE4 = 1321905599;                   // 2^61
constexpr int kE5 = 1466040222;                   // 2^70
constexpr int kE6 = 2646306;                      // 2^70
}  // namespace fxc

// sin and cos of (pi/32) (k + f) in Q62, 0 <= k <= 64 and f in Q63, |f| <= 1/2, with an
// error of a few 2^-60: Taylor polynomials of the remainder (their inner terms, which
// reach the result by powers of a square below 2^-9, in 32 bits), the angle-
// addition formulas.
__device__ __forceinline__ void fx_sincos_at(unsigned k, long long f, const MathTables* t, long long* sn, long long* cs) {
    const Fx F = fx(f);
    const long long z = fx_mad(F, F, 0);                                      // f^2 in Q62
    const Fx Z = fx(z);
    const int z32 = (int)(z >> 30);                                           // Q32, < 2^30
    const int i7 = fxc::kS7 - __mulhi(z32, fxc::kS9);
    const int i5 = fxc::kS5 - (__mulhi(z32, i7) >> 8);
    const long long i3 = fxc::kS3 - (((long long)z32 * i5) >> 12);
    const long long P = fxc::kS1 - (fx_mad(Z, fx(i3), 0) >> 6);               // Q66
    const Fx sr = fx(fx_mad(F, fx(P), 0));                                    // sin r in Q65
    const int i6 = fxc::kC6 - __mulhi(z32, fxc::kC8);
    const long long i4 = fxc::kC4 - (((long long)z32 * i6) >> 10);
    const long long i2 = fxc::kC2 - (fx_mad(Z, fx(i4), 0) >> 8);              // Q70
    const Fx nc = fx(-(fx_mad(Z, fx(i2), 0) >> 3));                           // -(1 - cos r) in Q65
    const long long Sk = t->sq[k], Ck = t->cq[k];
    const Fx S = fx(Sk), C = fx(Ck);
    *sn = Sk + (fx_mad(C, sr, fx_mad(S, nc, 0)) >> 1);                        // sums in Q63
    *cs = Ck + ((fx_mad(C, nc, 0) - fx_mad(S, sr, 0)) >> 1);
}

// sin and cos of phi in Q62, |phi| < 4: phi in units of pi/32, nearest table entry.
__device__ __forceinline__ void fx_sincos(double phi, const MathTables* t, long long* sn, long long* cs) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(phi);
    const unsigned long long X = fx_magnitude(b, 2);                          // |phi| in Q61
    const unsigned long long U = __umul64hi(X, fp64tab::kTwoOverPiQ64);       // |phi| 32/pi in Q57
    const unsigned k = (unsigned)((U + (1ull << 56)) >> 57);
    const long long f = (long long)((U - ((unsigned long long)k << 57)) << 6);   // Q63, |f| <= 1/2
    long long sv;
    fx_sincos_at(k > 64u ? 64u : k, f, t, &sv, cs);
    *sn = (long long)b < 0 ? -sv : sv;
}

// sqrt(a b) in Q62 and the product itself in Q62 for a, b in Q62 within (2^-17,
// 1]: the product of the normalised factors, an FP32 reciprocal root y of its
// leading 32 bits (relative error below 2^-21), and sqrt x = x y (1 + e/2 + 3 e^2 /
// 8 + ...) with e = 1 - x y^2 from exact products: cut off below 2^-64.
__device__ __forceinline__ long long fx_sqrt_product(long long a, long long b, long long* product) {
    const int la = __clzll(a) & 63, lb = __clzll(b) & 63;                     // 1 .. 19
    const unsigned long long p = __umul64hi((unsigned long long)a << la, (unsigned long long)b << lb);
    const int d = la + lb;                                                    // a b = p 2^(4 - d) 2^-64, p >= 2^62
    *product = (long long)(p >> ((d - 2) & 63));
    const unsigned long long x = p >> (d & 1);                                // Q64, in [1/8, 1)
    const int e2 = d >> 1;                                                    // sqrt(a b) = sqrt(x) 2^(2 - e2), e2 >= 1
    const unsigned xh = (unsigned)(x >> 32), xl = (unsigned)x;
    const float y = rsqrtf((float)xh * 2.3283064365386963e-10f);              // [1, 2.83)
    const unsigned yb = __float_as_uint(y);
    const unsigned Y = ((yb & 0x7FFFFFu) | 0x800000u) << (((yb >> 23) - 127u + 6u) & 31u);   // Q29
    const unsigned long long Y2 = (unsigned long long)Y * Y;                  // Q58
    const long long e = (long long)((1ull << 58) - __umul64hi(x, Y2));        // Q58, |e| < 2^38
    const int e16 = (int)(e >> 16);                                           // Q42
    const long long c = (e >> 1) + ((3 * (((long long)e16 * e16) >> 26)) >> 3);
    // s0 = x y in Q62, s = s0 (1 + c)
    const long long s0 = (long long)((((unsigned long long)xh * Y) << 1) + (((unsigned long long)xl * Y) >> 31));
    const unsigned long long s = (unsigned long long)(s0 + fx_mad(fx(s0), fx(c << 6), 0));   // Q62 x Q64 -> Q62
    return (long long)((s << 1) >> ((e2 - 1) & 63));
}

// Whether fx_basis holds its accuracy for these angles: |phi| < 4 and |cos thK|,
// |cos thmu| < 1 - 2^-17, so that sin^2 = 1 - cos^2 >= 2^-16 and its fixed-point
// error (2^-60 absolute) stays below 2^-44 relative.  Outside (about 1.5e-5 of
// uniformly distributed angles, and invalid |cos| > 1 or NaN) the caller uses the
// FP64 basis.
__device__ __forceinline__ bool fx_angles_ok(double ck, double cl, double phi) {
    constexpr double kMaxCos = 1.0 - 0x1p-17;
    return abs_below(ck, kMaxCos) && abs_below(cl, kMaxCos) && abs_below(phi, 4.0);
}

// |x| < 1.75: a basis value (or product) that Q62 holds, with room; false for NaN.
__device__ __forceinline__ bool fits_q62(double x) {
    return ((int)((unsigned long long)__double_as_longlong(x) >> 32) & 0x7FFFFFFF) < 0x3FFC0000;
}

// Ten products of the helicity angles in Q62, a basis of the f'_k (angular.cuh) that takes
// one product less each.  Absolute error a few 2^-60; in the four with the square root q of
// sk2 sl2 also those factors' last places times (sk2 + sl2) / (2 q), up to 2^-55 near |cos| = 1:
//   g = {sl2, sk2, G, G cp^2, G sp cp, f'_4, f'_5, f'_7, f'_8, f'_9},  G = sk2 sl2 (sk2 =
//   sin^2 thK, sl2 = sin^2 thmu, cp = cos phi, sp = sin phi);
//   f'_0 = sl2 - G, f'_1 = sk2 - G cp^2, f'_2 = sk2 - G + G cp^2, f'_3 = G sp cp, f'_6 = sl2.
__device__ __forceinline__ void fx_basis(double ck, double cl, double phi, const MathTables* t, long long g[10]) {
    long long sp, cp;
    fx_sincos(phi, t, &sp, &cp);
    const unsigned long long cb = (unsigned long long)__double_as_longlong(ck);
    const unsigned long long lb = (unsigned long long)__double_as_longlong(cl);
    const unsigned long long ca = fx_magnitude(cb, 0), la = fx_magnitude(lb, 0);   // |cos| in Q63, < 1
    const long long CKv = (long long)cb < 0 ? -(long long)(ca >> 1) : (long long)(ca >> 1);      // Q62
    const long long CLv = (long long)lb < 0 ? -(long long)(la >> 1) : (long long)(la >> 1);
    // 1 - c^2 = (1 - |c|) (1 + |c|) in Q62
    const long long sk2 = (long long)__umul64hi((1ull << 63) - ca, (1ull << 63) + ca);
    const long long sl2 = (long long)__umul64hi((1ull << 63) - la, (1ull << 63) + la);
    long long G;
    const long long q = fx_sqrt_product(sk2, sl2, &G);
    const Fx SP = fx(sp), CP = fx(cp), CK = fx(CKv), CL = fx(CLv), SL = fx(sl2);
    g[0] = sl2;
    g[1] = sk2;
    g[2] = G;
    const Fx gc = fx(fx_q62(fx(G), CP));
    g[3] = fx_q62(gc, CP);
    g[4] = fx_q62(gc, SP);
    const Fx b = fx(fx_q62(fx(q), CL));
    g[7] = fx_q62(b, CP);
    g[8] = fx_q62(b, SP);
    g[5] = fx_q62(fx(g[7]), CK);
    g[6] = fx_q62(fx(g[8]), CK);
    g[9] = fx_q62(CK, SL);
}

// A linear function of t, y = c - t g with g = rate (inv + inv_lo), in fixed point: part of
// a segment's record (ipa_internal.cuh).  y has ysh fraction bits (|y| 2^ysh < 2^60), t is taken
// with `top`, |t| < 2^(top - 1); g is carried to 2^-61 of itself, so that the error of y does not
// grow with t.  ok = 0 where some |y| could reach 65000 (or is NaN).  Compiled without FMA
// contraction.
__device__ inline FxExp fx_line_setup(double rate, double inv, double inv_lo, double c, double t_most) {
    FxExp s = {0, 0, 0, 2, 32, 0, 0};
    const double g = rate * inv, g_lo = fma(rate, inv, -g) + rate * inv_lo;
    const int e = (int)((__double_as_longlong(t_most) >> 52) & 0x7FF) - 1022;      // t_most < 2^e
    if (!(t_most > 0.0) || e > 60 || e < -60) return s;
    const double ag = abs_bits(g), m = ag * __longlong_as_double((long long)(e + 1023) << 52) + abs_bits(c);
    if (!(m < 65000.0)) return s;                        // beyond the doubles' range (and NaN)
    const int ey = (int)((__double_as_longlong(m) >> 52) & 0x7FF) - 1022;          // m < 2^ey
    s.top = e + 1;
    s.ysh = 60 - (ey > 6 ? ey : 6);
    // c 2^ysh and g 2^(ysh + top + 1), both below 2^62
    s.c = fx_signed(c, 63 - s.ysh);
    const Fx gf = fx(fx_signed(g, 62 - s.ysh - s.top) + fx_signed(g_lo, 62 - s.ysh - s.top));
    s.gh = gf.h;
    s.gl = gf.l;
    s.ok = 1;
    return s;
}

// For fx_exp: 2 e^{-Gamma tau + c_exp} = 2^(y/64), y = 64 (1 + (Gamma mu + c_exp) / ln2) - t 64 Gamma / ln2.
__device__ inline FxExp fx_exp_setup(double Gamma, double mu, double c_exp, double t_most) {
    return fx_line_setup(Gamma, 92.33248261689366, 1.3027375194195861e-15, 64.0 + (Gamma * mu + c_exp) * 92.33248261689366, t_most);
}
// For fx_phase: Dm tau - ph0 in units of pi/32.
__device__ inline FxExp fx_phase_setup(double Dm, double mu, double ph0, double t_most) {
    return fx_line_setup(neg_bits(Dm), 10.185916357881302, -6.297176536058395e-16, neg_bits(Dm * mu + ph0) * 10.185916357881302, t_most);
}

// 2^(y / 64) for y in fixed point with ysh fraction bits, as a double: table and Taylor
// polynomial of degree 6 in the fraction.  *x: the power of two (the result is normal
// for -1015 <= x < 1015, else unspecified).
__device__ __forceinline__ double fx_exp2(long long y, int ysh, const MathTables* mt, int* x) {
    const int k = (int)(y >> ysh);
    const unsigned long long f = (unsigned long long)y << ((64 - ysh) & 63);   // fraction, Q64
    const unsigned f32 = (unsigned)(f >> 32);
    const Fx F = fx((long long)(f >> 2));                                     // Q62
    const unsigned i5 = (unsigned)fxc::kE5 + __umulhi(f32, (unsigned)fxc::kE6);
    const unsigned i4 = (unsigned)fxc::kE4 + (__umulhi(f32, i5) >> 9);
    const long long i3 = fxc::kE3 + (long long)(((unsigned long long)f32 * i4) >> 9);
    const long long i2 = fxc::kE2 + (fx_mad(F, fx(i3), 0) >> 6);
    const long long i1 = fxc::kE1 + (fx_mad(F, fx(i2), 0) >> 5);
    const Fx p = fx(fx_mad(F, fx(i1), 0));                                    // 2^(f/64) - 1 in Q67
    const long long e = mt->eq[k & 63];                                       // Q62
    const unsigned long long v = (unsigned long long)(e + (fx_mad(fx(e), p, 0) >> 3));   // [2^62, 2^63]
    *x = k >> 6;
    return __longlong_as_double((long long)(((v - (1ull << 62) + 512ull) >> 10) +
                                            ((unsigned long long)(unsigned)(*x + 1023) << 52)));
}

// 2 e^{-Gamma tau + Gamma^2 sigma^2 / 2} (fx_exp_setup) at t, T = fx(fx_signed(t, s.top)).
// Relative error before the last rounding: ln2 / 64 times the error of y, two units of 2^-ysh
// (ysh = 54 where |y| < 64 throughout the range, 44 at 65000) and the rounding of c as a double
// (2^-47 for |c| < 128, as with mu near 0): 2^-53.5 for the usual ranges, 2^-50 at the widest.
// *ok is cleared where the result lies outside its range (the caller checks fx_in_range).
__device__ __forceinline__ double fx_exp(Fx T, const FxExp& s, const MathTables* mt, bool* ok) {
    int x;
    const double v = fx_exp2(s.c - fx_mad(T, Fx{s.gh, s.gl}, 0), s.ysh, mt, &x);
    *ok = *ok && (unsigned)(x + 1015) < 2030u;
    return v;
}
__device__ __forceinline__ bool fx_in_range(double t, int top) {
    return (int)((unsigned)((unsigned long long)__double_as_longlong(t) >> 52) & 0x7FFu) - 1022 < top;
}

// sin and cos (Q62) of the phase of fx_phase_setup at t.
__device__ __forceinline__ void fx_phase(Fx T, const FxExp& s, const MathTables* mt, long long* sn, long long* cs) {
    const unsigned long long y = (unsigned long long)(s.c - fx_mad(T, Fx{s.gh, s.gl}, 0));
    const unsigned long long up = y + (1ull << ((s.ysh - 1) & 63));
    const unsigned k = (unsigned)((long long)up >> (s.ysh & 63));
    fx_sincos_at(k & 63u, (long long)((up << ((64 - s.ysh) & 63)) ^ (1ull << 63)) >> 1, mt, sn, cs);
}

// e^a for -705 <= a <= 0: |a| in units of ln2/64, its fixed point following its
// exponent (error before the last rounding below 2^-54 for |a| < 32, |a| 2^-59 beyond).
__device__ __forceinline__ double fx_exp_neg(double a, const MathTables* mt) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(a);
    const int E = (int)((b >> 52) & 0x7FFull) - 1023;
    const int top = E + 1 > 2 ? E + 1 : 2;
    const long long T = (long long)fx_magnitude(b, top);   // up to 2^63 - 1
    constexpr Fx kInv = {774541002, 1460010031};        // 64 / ln2 in 2^55
    int x;
    return fx_exp2(fx_mad(fx(-T), kInv, 0), (54 - top) & 63, mt, &x);
}

// erfcx(x) = exp(x^2) erfc(x) for 0 <= x <= 6.25 (the pieces of erfcx_poly); larger x,
// infinities and NaN are evaluated as 6.25.
__device__ __forceinline__ double fx_erfcx(double x, const MathTables* t) {
    using namespace fp64tab;
    long long b = __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll;
    b = b > 0x4019000000000000ll ? 0x4019000000000000ll : b;
    const unsigned long long X = fx_magnitude((unsigned long long)b, 3);      // Q60
    int k = (int)((X + (1ull << 58)) >> 59);                                  // nearest piece centre k/2
    k = k > kErfcxPieces - 1 ? kErfcxPieces - 1 : k;
    const Fx U = fx((long long)((X - ((unsigned long long)k << 59)) << 4));   // Q64, |u| <= 1/4
    const long long* c = t->exq + k * kErfcxCoeffs;
    long long v = c[kErfcxCoeffs - 1];
#pragma unroll
    for (int i = kErfcxCoeffs - 2; i >= 0; --i) v = fx_mad(fx(v), U, c[i]);   // |v| < 1.5 in Q62
    return fx_to_double(v, 0);
}

// log x for 2^-126 <= x < 2^127 (positive and normal, the caller checks) in Q56: x = 2^e m,
// r = m c_j - 1 with the table's c_j (log_fast), |r| <= 2^-8, log1p's series to r^7, its
// terms from r^4 on in 32 bits.  Error below (2 + |e| / 3) 2^-56, the second part ln 2's
// rounding: 2^-55 at e = 0, 2^-50.5 at |e| = 126, and always below 2^-55 of |log x| + 1.
__device__ __forceinline__ long long fx_log(double x, const MathTables* t) {
    const long long b = __double_as_longlong(x);
    const int e = (int)(b >> 52) - 1023;
    const int j = (int)((b >> 45) & 127);
    const long long m = (long long)(((unsigned long long)b << 10 & 0x3FFFFFFFFFFFFFFFull) | 0x4000000000000000ull);  // Q62
    const long long cb = __double_as_longlong(t->linv[j]);                    // in [1/2, 1)
    const long long c = (long long)(((unsigned long long)cb << 9 & 0x1FFFFFFFFFFFFFFFull) | 0x2000000000000000ull);  // Q62
    const long long r = -fx_mad(fx(-m), fx(c), 1ll << 60);                    // Q60 (m < 2^63: negated for fx)
    const Fx R = fx(r << 10);                                                 // Q70
    const int r32 = R.h;                                                      // Q38, |r32| <= 2^30
    const int i6 = 357913941 - (__mulhi(r32, 306783378) >> 6);                // 1/6 - r/7 in 2^31
    const int i5 = 429496730 - (__mulhi(r32, i6) >> 6);
    const int i4 = 536870912 - (__mulhi(r32, i5) >> 6);
    const long long i3 = 1537228672809129301ll - (((long long)r32 * i4) >> 7);   // 1/3 - ... in Q62
    const long long i2 = (1ll << 61) - (fx_mad(R, fx(i3), 0) >> 6);           // Q62
    const Fx r2 = fx(fx_mad(R, R, 0));                                        // r^2 in Q76
    const long long l = r - (fx_mad(r2, fx(i2), 0) >> 14);                    // log1p r in Q60
    return (long long)e * fp64tab::kLn2Q56 + t->lq[j] + (l >> 4);
}

}  // namespace ipa
