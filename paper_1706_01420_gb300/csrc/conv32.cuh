// FP32 copies of the convolved decay exponentials, with error bounds, for the
// FP32 decision filters of the generators of the tagged and the phi_s models:
//   H, L = g(tau; Gamma_H), g(tau; Gamma_L),  Cr + i Ci = g(tau; Gamma - i Dm),
// g(tau; z) = 1/2 exp(-z tau + z^2 sigma^2 / 2) erfc((z sigma^2 - tau) / (sqrt2 sigma)).
// Away from the resolution peak (every erfc within 1.2e-9 of 2) they are
// exponentials; near it they take erfcf and the Faddeeva function by
// Weideman's rational approximation with N = 16 in FP32 (relative error
// below 1e-6 in FP32 arithmetic over 0 <= Re z <= 8, Im z >= 0, measured against
// scipy's wofz; 3e-6 is charged).  The bounds are of the worst case with factors
// to spare (the errors met over 1.2e6 candidates of 12 parameter points stay below
// 6 % of them) and still leave FP64 only one phi_s candidate in 5000 and one
// tagged candidate in 10^5.
#pragma once

#include "accept_reject.cuh"

namespace ipa {

// e^{off - x tau} in base 2.
struct Exp32 {
    float x, off;
};

struct Conv32 {
    Exp32 H, L, C;       // the exponentials of 2 g / 2 (C: the oscillation's amplitude)
    float uH0, uL0, uC0; // x sigma^2
    float k_z, k_g, beta;
    float d;             // t_lo - mu
    float near;          // tau above it: every erfc argument is below -4.3
    float x, off;        // the largest |x| and |off| of the three exponentials
};

constexpr float kMaxArg = 99.0f;     // |base-2 exponent| where the FP32 exponential keeps its accuracy
constexpr double kLog2e = 1.44269504088896340736;

__device__ __forceinline__ Exp32 exp32_of(double x, double off) {
    return Exp32{(float)(x * kLog2e), (float)(off * kLog2e)};
}

// 2^x (relative error below 2^-22; 0 below -126)
__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Bound of the relative error of exp2f(off - x tau), tau off by dtau: the
// argument is off by |x| dtau and by four roundings of terms no larger than
// |x tau| + |off|; exp2f adds 2 ulp; a factor 2 and 1e-6 to spare.
__device__ __forceinline__ float exp32_err(float x, float off, float tau, float dtau) {
    return 2.0f * (0.7f * (x * dtau + kUlp1 * fmaf(x, fabsf(tau), off)) + 2.5e-7f) + 1.0e-6f;
}

// Bound of the error of tau = fmaf(u32, span, d): the uniform's, the span's and
// d's roundings and the sum's, |u span| <= |tau| + |d|, with a factor above 1.3 to spare.
__device__ __forceinline__ float tau32_err(float tau, float d, float span) {
    return kUlp1 * (fabsf(tau) + fabsf(d)) + 9.4e-10f * span;
}

// C: a record with the fields of TagConsts read below (TagConsts, PhisConsts);
// d = t_lo - mu, span = t_hi - t_lo.
template <class C>
__device__ inline Conv32 conv32_of(const C& c, double d, double span) {
    constexpr double kLn2d = 0.69314718055994530942;
    Conv32 v;
    v.d = (float)d;
    v.H = exp32_of(c.GH, c.cH2 - kLn2d);
    v.L = exp32_of(c.GL, c.cL2 - kLn2d);
    v.C = exp32_of(c.Gamma, c.cC2 - kLn2d);
    v.uH0 = (float)c.uH0;
    v.uL0 = (float)c.uL0;
    v.uC0 = (float)c.uC0;
    v.k_z = (float)c.k_z;
    v.k_g = (float)c.k_g;
    v.beta = (float)c.beta;
    const double top = fmax(fmax(c.uH0, c.uL0), c.uC0);
    v.near = c.k_z > 0.0 ? (float)(top + 4.3 / c.k_z) * 1.000001f + 1.0e-6f * ((float)span + fabsf(v.d)) : INFINITY;
    v.x = fmaxf(fmaxf(fabsf(v.H.x), fabsf(v.L.x)), fabsf(v.C.x));
    v.off = fmaxf(fmaxf(fabsf(v.H.off), fabsf(v.L.off)), fabsf(v.C.off));
    return v;
}

// The phase Dm tau - ph0 in half turns, reduced to [-1, 1], for tau = tau0 + u
// span with u the 32-bit uniform word: u span Dm / pi in fixed point (2^-24 of a
// half turn times 2^-32), so that a range of many turns costs no accuracy.
// Error below 2^-25 (the step) + 2^-32 |K| (the uniform's lower bits) + 2^-24
// (the float) half turns: kPhaseErr radians with a factor 2 to spare.  |K| <
// 128 half turns over the range (ok), else the phase is not established.
struct Phase32 {
    int32_t step;        // K 2^24, K = span Dm / pi
    int64_t base;        // (Dm tau0 - ph0) / pi modulo 2, in 2^-56
    bool ok;
};
constexpr float kPhaseErr = 1.5e-6f;

__device__ inline Phase32 phase32_of(double Dm, double ph0, double tau0, double span) {
    constexpr double kInvPi = 0.31830988618379067154;
    const double K = span * Dm * kInvPi;
    const double b = (Dm * tau0 - ph0) * kInvPi;
    Phase32 p;
    p.ok = fabs(K) < 127.0 && fabs(b) < 1.0e6;
    p.step = p.ok ? (int32_t)rint(K * 16777216.0) : 0;
    const double r = p.ok ? b - 2.0 * rint(0.5 * b) : 0.0;      // [-1, 1]
    p.base = (int64_t)(r * 72057594037927936.0);
    return p;
}
__device__ __forceinline__ float phase32(const Phase32& p, uint32_t u) {
    const uint64_t v = (uint64_t)p.base + (uint64_t)((int64_t)p.step) * u;   // 2^-56 half turns, modulo 2^64
    return (float)(int32_t)(uint32_t)(v >> 25) * 4.656612873077393e-10f;     // bits 25..56: modulo 2, in 2^-31
}

// The exponentials alone; ok: tau lies above the peak and every bound holds.
struct Far32 {
    float H, L, C, err;  // err: relative error bound of the exponentials
    bool ok;
};
__device__ __forceinline__ Far32 conv32_far(const Conv32& v, float tau, float dtau) {
    const float aH = fmaf(-v.H.x, tau, v.H.off), aL = fmaf(-v.L.x, tau, v.L.off), aC = fmaf(-v.C.x, tau, v.C.off);
    Far32 g;
    g.H = exp2f(aH);
    g.L = exp2f(aL);
    g.C = exp2f(aC);
    g.err = exp32_err(v.x, v.off, tau, dtau);
    g.ok = tau > v.near && fabsf(aH) <= kMaxArg && fabsf(aL) <= kMaxArg && fabsf(aC) <= kMaxArg && g.err <= 1.0e-3f;
    return g;
}

// Weideman's coefficients for N = 16, L = 2^(-1/4) sqrt(16) (faddeeva.cuh gives the method).
__device__ const float kWeid16[16] = {
    1.748395886e+00f,  1.362240822e+00f,  8.864478302e-01f, 4.692909009e-01f,  1.912417267e-01f,  5.182240243e-02f,
    3.682567317e-03f,  -3.881015189e-03f, -1.527659740e-03f, 8.703158428e-05f, 2.107105640e-04f,  2.170986793e-05f,
    -2.734640462e-05f, -5.584233411e-06f, 3.981287575e-06f, 9.939322536e-07f};
constexpr float kWeid16L = 3.363585661014858f;

__device__ __forceinline__ void faddeeva32(float x, float y, float* wr, float* wi) {
    const float dr = kWeid16L + y;
    const float inv = __frcp_rn(fmaf(dr, dr, x * x));
    const float er = dr * inv, ei = x * inv;
    const float nr = kWeid16L - y;
    const float zr = fmaf(nr, er, -(x * ei)), zi = fmaf(nr, ei, x * er);
    float pr = kWeid16[15], pi = 0.0f;
#pragma unroll
    for (int k = 14; k >= 0; --k) {
        const float t = fmaf(pr, zr, fmaf(-pi, zi, kWeid16[k]));
        pi = fmaf(pr, zi, pi * zr);
        pr = t;
    }
    const float tr = fmaf(2.0f, fmaf(pr, er, -(pi * ei)), 0.5641895835f);
    const float ti = 2.0f * fmaf(pr, ei, pi * er);
    *wr = fmaf(tr, er, -(ti * ei));
    *wi = fmaf(tr, ei, ti * er);
}

// The four functions at tau; H, L and C (C >= |Cr + i Ci|, at least the larger of
// its two terms) are within err (relative), Cr and Ci within err C.  err = inf
// where the bounds are not established.
struct Time32 {
    float H, L, C, Cr, Ci, err;
};

__device__ __forceinline__ Time32 conv32(const Conv32& v, float tau, float dtau, float phase, bool phase_ok) {
    Time32 g;
    const Far32 f = conv32_far(v, tau, dtau);
    float sn, cn;
    sincospif(phase, &sn, &cn);
    g.H = f.H;
    g.L = f.L;
    g.C = f.C;
    g.Cr = f.C * cn;
    g.Ci = f.C * sn;
    g.err = f.ok && phase_ok ? 2.0f * (f.err + kPhaseErr) : INFINITY;
    if (f.ok || !phase_ok || !(f.err <= 1.0e-3f)) return g;
    // near the peak: z = (x sigma^2 - tau) k_z is off by dz; erfcf adds 4 ulp, and the
    // argument error enters through |erfc'| / erfc <= z + sqrt(z^2 + 2) (z >= 0;
    // Abramowitz and Stegun 7.1.13) or <= 2/sqrt(pi) (z < 0)
    const float zH = (v.uH0 - tau) * v.k_z, zL = (v.uL0 - tau) * v.k_z, a = (v.uC0 - tau) * v.k_z;
    const float top = fmaxf(fmaxf(fabsf(v.uH0), fabsf(v.uL0)), fabsf(v.uC0));
    const float zm = fmaxf(fmaxf(zH, zL), a), za = fmaxf(fmaxf(fabsf(zH), fabsf(zL)), fabsf(a));
    const float dz = v.k_z * (dtau + kUlp1 * (top + fabsf(tau))) + kUlp2 * za;
    const float sens = zm > 0.0f ? zm + sqrtf(fmaf(zm, zm, 2.0f)) : 1.2f;
    const float rel = 2.0f * (1.1f * sens * dz + 2.0e-6f) + f.err;
    const float gr = tau * tau * v.k_g;
    // |w'| <= 2/sqrt(pi) in the upper half plane
    const float gx = expf(-gr), egx = 2.0f * (2.0f * fabsf(tau) * v.k_g * dtau + kUlp2 * gr) + 2.0e-6f;
    if (!(v.k_z > 0.0f) || !(zm <= 7.0f) || !(rel <= 1.0e-2f) || !(egx <= 1.0e-2f) || !(gr <= 80.0f) || !(fabsf(v.beta) <= 8.0f) ||
        !(fabsf(f.H) <= 1.0e30f) || !(fabsf(f.L) <= 1.0e30f) || !(fabsf(f.C) <= 1.0e30f)) {
        g.err = INFINITY;
        return g;
    }
    g.H = 0.5f * f.H * erfcf(zH);
    g.L = 0.5f * f.L * erfcf(zL);
    float wr, wi;
    const bool ap = a >= 0.0f;
    faddeeva32(fabsf(v.beta), fabsf(a), &wr, &wi);
    if ((v.beta >= 0.0f) != ap) wi = -wi;            // w at +beta for a >= 0 and at -beta for a < 0
    const float hx = 0.5f * gx;
    const float e = ap ? 0.0f : f.C;
    g.Cr = ap ? hx * wr : fmaf(f.C, cn, -hx * wr);
    g.Ci = ap ? hx * wi : fmaf(f.C, sn, -hx * wi);
    g.C = e + hx;
    // the oscillation is within e (err + the phase's) + hx (egx + 1.2 dz + 3e-6 and the error of beta)
    g.err = fmaxf(rel, 2.0f * (f.err + kPhaseErr) + 2.0f * (egx + 1.2f * (dz + kUlp1 * fabsf(v.beta)) + 6.0e-6f));
    return g;
}

}  // namespace ipa
