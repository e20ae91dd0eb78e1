// The Faddeeva function w(z) = exp(-z^2) erfc(-i z) in the upper half plane,
// for the decay-time terms of the tagged model: the convolution of an
// oscillating exponential e^{-(Gamma - i Dm) t} with a Gaussian is a complex
// erfc, which Sec. 2 and the symbolic-programming section of the paper
// evaluate through w(z).
//
// Method: Weideman's rational approximation (J.A.C. Weideman, "Computation of
// the complex error function", SIAM J. Numer. Anal. 31 (1994) 1497).  For
// Im z > 0, w(z) = (i/pi) int e^{-t^2} / (z - t) dt.  With t = L tan(theta/2),
// e^{-t^2} (L^2 + t^2) = sum_n a_n e^{i n theta} (even in theta) and
// e^{i theta} = (L + i t) / (L - i t); integrating each term by residues
// (closing the contour above for n >= 0, below for n < 0) gives
//   w(z) = 1 / (sqrt(pi) (L - i z)) + 2 sum_{n>=1} a_n Z^{n-1} / (L - i z)^2,
//   Z = (L + i z) / (L - i z),
// truncated at n = N = 40 with L = 2^(-1/4) sqrt(N).  The coefficients are
// generated in 60-digit arithmetic (gen_fp64_tables.py).  |Z| <= 1 in the closed
// upper half plane, and |L - i z| >= L keeps every division away from zero.
//
// The coefficients are real, so p(Z) = sum a_k Z^k takes two real products per
// step instead of four:
//   b_k = a_k + 2 Re Z b_{k+1} - |Z|^2 b_{k+2},  p = a_0 + Z b_1 - |Z|^2 b_2.
// The recurrence runs on the integer pipe at the scale that the sums allow:
// b_39 .. b_24 (below 2^-27.5) as 32-bit numbers in Q58, b_23 .. b_8 (below 0.45)
// in Q62, b_7 .. b_1 (|b_k| <= sum_{j >= k} (j - k + 1) |a_j| < 42) in Q57.  An
// error at step k reaches p with a factor up to k + 1 (Z near +-1); with these
// scales the sum stays below 2^-51, and it reaches w divided by |L - i z|^2 / 2 >=
// 14.  Measured: 2.7e-16 rms and 1.5e-15 at worst over 0 <= x < 8, 0 <= y <
// 1000, all of it from the FP64 parts (1/d, Z, the combination).  The four-product
// Horner sum with full 64-bit products took five times the instructions:
// 1e6 tagged events 185 us with it, 131 us with this and the cheaper exponentials.
#pragma once

#include <math.h>

#include "fp64_tables.cuh"
#include "fast_fixed.cuh"

namespace ipa {

// The part of v within the 32-bit range.
__device__ __forceinline__ int clamp_q31(long long v) {
    return v > 0x7FFFFFFFll ? 0x7FFFFFFF : (v < -0x7FFFFFFFll ? -0x7FFFFFFF : (int)v);
}

// w(x + i y) for y >= 0: about 25 FP64 operations and the fixed-point sum.  It is
// evaluated at |x| and conjugated for x < 0 (w(-conj z) = conj w(z)), so that
// symmetry holds bit for bit.
__device__ __forceinline__ void faddeeva_uhp(double xs, double y, double* wr, double* wi) {
    using namespace fp64tab;
    const double x = abs_bits(xs);
    // d = L - i z = (L + y) - i x;  1/d = ((L + y) + i x) / |d|^2
    const double dr = kWeidL + y;
    const double d2 = fma(dr, dr, x * x);
    double inv = rcp_newton(d2);                                // to about 6e-14; one more step
    if (!above(d2, 4e37)) inv = fma(inv, fma(-d2, inv, 1.0), inv);
    const double er = dr * inv, ei = x * inv;
    // Z = (L + i z) / d = ((L - y) + i x) / d
    const double nr = kWeidL - y;
    const double Zr = fma(nr, er, -(x * ei)), Zi = fma(nr, ei, x * er);
    // p(Z) = sum a_k Z^k = a_0 + Z b_1 - |Z|^2 b_2, b_k = a_k + 2 Re Z b_{k+1} - |Z|^2 b_{k+2}
    const long long R64 = fx_signed(Zr, 1), I64 = fx_signed(Zi, 1);                           // Q62
    const long long S64 = (long long)(((unsigned __int128)((__int128)R64 * R64) + (unsigned __int128)((__int128)I64 * I64)) >> 62);
    const int R30 = clamp_q31(R64 >> 31), S30 = -clamp_q31(S64 >> 31);                        // 2 Re Z in Q30, -|Z|^2 in Q31
    int c1 = 0, c2 = 0;                                                                       // Q58, below 2^31
#pragma unroll 4
    for (int k = kWeidN - 1; k >= 24; --k) {
        const long long m = (long long)c1 * R30 + (((long long)c2 * S30) >> 1);
        c2 = c1;
        c1 = (int)(kWeidAQ59[k] >> 1) + (int)(m >> 30);
    }
    const Fx R = fx(R64), S = fx(-S64);
    long long b1 = (long long)c1 << 4, b2 = (long long)c2 << 4;                               // Q62
#pragma unroll 2
    for (int k = 23; k >= 8; --k) {
        const Fx f1 = fx(b1);
        const long long m = (fx_mad(f1, R, 0) << 1) + fx_mad(fx(b2), S, 0);                   // Q60
        b2 = b1;
        b1 = (kWeidAQ59[k] << 3) + (long long)((unsigned long long)m << 2);
    }
    b1 >>= 5;                                                                                 // Q57, below 42
    b2 >>= 5;
#pragma unroll 2
    for (int k = 7; k >= 1; --k) {
        const long long m = (fx_mad(fx(b1), R, 0) << 1) + fx_mad(fx(b2), S, 0);               // Q55
        b2 = b1;
        b1 = (kWeidAQ59[k] >> 2) + (long long)((unsigned long long)m << 2);
    }
    const Fx B1 = fx(b1);
    const long long qr = (kWeidAQ59[0] >> 2) + (long long)((unsigned long long)(fx_mad(B1, R, 0) + fx_mad(fx(b2), S, 0)) << 2);
    const long long qi = (long long)((unsigned long long)fx_mad0(B1, fx(I64), 0) << 2);   // 0 for Im Z = 0
    const double pr = fx_to_double(qr, 5), pi = fx_to_double(qi, 5);                          // Q57
    // w = (2 p / d + 1/sqrt(pi)) / d
    const double tr = fma(2.0, fma(pr, er, -(pi * ei)), kInvSqrtPi);
    const double ti = 2.0 * fma(pr, ei, pi * er);
    *wr = fma(tr, er, -(ti * ei));
    const double wim = fma(tr, ei, ti * er);
    *wi = negative(xs) ? neg_bits(wim) : wim;
}

// w(z) anywhere: the upper half plane directly, the lower by the reflection
// w(z) = 2 exp(-z^2) - w(-z) (library exp and sincos; it overflows where
// exp(-z^2) does).
__device__ __forceinline__ void faddeeva(double x, double y, double* wr, double* wi) {
    if (!(y < 0.0)) {
        faddeeva_uhp(x, y, wr, wi);
        return;
    }
    double ur, ui;
    faddeeva_uhp(-x, -y, &ur, &ui);
    // exp(-z^2) = exp(y^2 - x^2) (cos(2xy) - i sin(2xy))
    const double m = 2.0 * exp((y - x) * (y + x));
    double s, c;
    sincos(2.0 * x * y, &s, &c);
    *wr = fma(m, c, -ur);
    *wi = fma(-m, s, -ui);
}

}  // namespace ipa
