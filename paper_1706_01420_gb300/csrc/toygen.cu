// Hot-path step a7: pseudo-experiment generation by accept-reject (Sec. 7).
//
// Sec. 7 of the paper draws curand uniforms per thread and keeps the events
// that pass an accept-reject test, with the event counts drawn on the host.
// Here the generator is Philox-4x32-10 (Salmon et al., SC'11) written out in
// this file, addressed by counters so that every candidate of every toy is a
// pure function of (seed, toy, candidate index):
//   key     = (seed lo32, seed hi32)
//   signal candidate j of toy k:  counters (j lo32, j hi32, k, c), c = 0, 1, 2
//     c = 0 -> (t = t_lo + u (t_hi - t_lo), u_t)
//     c = 1 -> (cos thK = 2u - 1, cos thmu = 2u - 1)
//     c = 2 -> (phi = pi (2u - 1), u_a)
//     kept iff u_t M_T < g(t - mu)  and (4D)  u_a M_Omega < A(Omega);
//   background event i of toy k:  counters (i lo32, i hi32, k, 4) -> (t, ck),
//                                 (.., 5) -> (cl, phi), always kept.
// Each 64-bit uniform is u = (((a << 32) | b) >> 11) + 1) 2^-53 from two
// 32-bit words, in (0, 1].  Candidates are built with correctly rounded
// multiplies and adds only (no contraction into FMA), so the event values are
// reproducible bit for bit on any IEEE machine.  A toy keeps its first n_sig
// accepted candidates in increasing j (accept_reject.cuh).
//
// Decisions first run in FP32 (this GPU's FP32 rate is 64 times its FP64
// rate): each test is evaluated with a per-candidate bound on its FP32 error,
// built from the documented accuracy of expf, exp2f, erfcf, sincospif and rsqrtf and
// the rounding of every input, and is decided in FP32 only when the uniform
// lies outside that band around the threshold.  Inside the band (about one
// candidate in 10^4), or wherever the bound is not established (a uniform or
// cosine near the end of its range, an exponent near over- or underflow), the
// FP64 test decides.  A decision is therefore always the FP64 test's; the
// FP32 pass only avoids evaluating it on clear cases.  Accepted candidates
// are regenerated from their counters and written with the exact FP64 values.
#include <math.h>

#include "accept_reject.cuh"
#include "consts.cuh"
#include "conv32.cuh"
#include "ipa_internal.cuh"
#include "philox.cuh"
#include "tagged.cuh"

namespace ipa {
namespace {

constexpr double kPi = 3.14159265358979323846;
constexpr double kSqrt2 = 1.41421356237309504880;
constexpr double k2OverSqrt6 = 0.81649658092772603273;
constexpr double k2OverSqrt3 = 1.15470053837925152902;

// A(Omega) = sum_k h_k f_k, evaluated as the oracle's definition (Sec. 4).
__device__ __forceinline__ double angular_pdf(const Consts& c, double ck, double cl, double phi) {
    const double sk = sqrt(1.0 - ck * ck), sl = sqrt(1.0 - cl * cl);
    double sp, cp;
    sincos(phi, &sp, &cp);
    double f[10];
    f[0] = ck * ck * sl * sl;
    f[1] = 0.5 * sk * sk * (1.0 - sl * sl * cp * cp);
    f[2] = 0.5 * sk * sk * (1.0 - sl * sl * sp * sp);
    f[3] = sk * sk * sl * sl * sp * cp;
    f[4] = kSqrt2 * sk * ck * sl * cl * cp;
    f[5] = -kSqrt2 * sk * ck * sl * cl * sp;
    f[6] = sl * sl / 3.0;
    f[7] = k2OverSqrt6 * sk * sl * cl * cp;
    f[8] = -k2OverSqrt6 * sk * sl * cl * sp;
    f[9] = k2OverSqrt3 * ck * sl * sl;
    double A = 0.0;
#pragma unroll
    for (int k = 0; k < 10; ++k) A += c.h[k] * f[k];
    return A;
}

__device__ __forceinline__ double time_pdf(const Consts& c, double t) {
    const double tau = t - c.mu;
    const double z = (c.Gs2 - tau) * c.k_z;
    return 0.5 * exp(-c.Gamma * tau + c.c_exp) * erfc(z);
}

// ---- FP32 decision filter ----
// Single-precision copies of what the tests read (set once per block).
struct Filter32 {
    float d;          // t_lo - mu
    float span;       // t_hi - t_lo
    float Gamma, c_exp, Gs2, k_z;
    float MT, MO;
    float h[10];
};

// +1: u_t M_T < g(t - mu) for sure; -1: not; 0: undecided (FP64 decides).
// Error bound per candidate (2^-22 ~ 2.4e-7 covers one float rounding with
// a factor 2 to spare): tau = d + u span carries
//   dtau <= 2^-22 (span + |tau| + |d|);
// the exponent a = -Gamma tau + c carries da <= |Gamma| dtau + 2^-21 (|Gamma tau| + |c|);
// expf adds 2 ulp; z = (Gamma sigma^2 - tau) k_z carries dz <= k_z (dtau + 2^-22
// |Gamma sigma^2|) + 2^-21 |z|; erfcf adds 4 ulp and the argument error enters
// through |erfc'(z)| / erfc(z) <= z + sqrt(z^2 + 2) (z >= 0; Abramowitz and
// Stegun 7.1.13) or <= 2/sqrt(pi) (z < 0, where erfc >= 1).
__device__ __forceinline__ int time_filter(const Filter32& f, uint32_t t_hi_word, uint32_t acc_hi_word) {
    const float tau = fmaf(u32of(t_hi_word), f.span, f.d);
    const float dtau = 2.384185791015625e-07f * (f.span + fabsf(tau) + fabsf(f.d));
    const float gt = f.Gamma * tau;
    const float arg = f.c_exp - gt;
    const float z = (f.Gs2 - tau) * f.k_z;
    if (!(fabsf(arg) <= 80.0f) || !(z <= 8.0f)) return 0;
    const float da = fabsf(f.Gamma) * dtau + 4.76837158203125e-07f * (fabsf(gt) + fabsf(f.c_exp));
    const float dz = f.k_z * (dtau + 2.384185791015625e-07f * fabsf(f.Gs2)) + 4.76837158203125e-07f * fabsf(z);
    const float sens = z > 0.0f ? z + sqrtf(fmaf(z, z, 2.0f)) : 1.2f;
    const float rel = 2.0f * (1.01f * da + 1.1f * sens * dz + 2.0e-6f) + 4.0e-6f;
    if (!(rel <= 1.0e-3f)) return 0;
    const float g = 0.5f * expf(arg) * erfcf(z);
    if (!(g >= 1.0e-30f) || !isfinite(g)) return 0;
    const float lhs = u32of(acc_hi_word) * f.MT;
    const float dl = lhs * 4.76837158203125e-07f + f.MT * 9.5367431640625e-07f;
    if (lhs + dl < g * (1.0f - rel)) return 1;
    if (lhs - dl > g * (1.0f + rel)) return -1;
    return 0;
}

// +1 / -1 / 0 for u_a M_Omega < A(Omega), from the words of calls 1 and 2.
// The cosines carry errors below 2.5e-7 and phi below 1.2e-6.  A sine (the
// square root of 1 - c^2, whose error is below 5e-7) is within 2.6e-7 of its
// value over itself for sin^2 >= 1e-5, and the sine and cosine of phi within
// 1.4e-6, so every f_k (constant factor included) is within ef = 5e-7 (1 / sin thK
// + 1 / sin thmu) + 2e-6, and |A32 - A| <= ef sum|h_k| + 6e-7 M_Omega <= 3 ef
// M_Omega (each max|f_k| >= 1/3): the band takes twice that.
__device__ __forceinline__ int angle_filter(const Filter32& f, const U4& b, const U4& e) {
    const float ck = fmaf(2.0f, u32of(b.x), -1.0f);
    const float cl = fmaf(2.0f, u32of(b.z), -1.0f);
    const float sk2 = fmaf(-ck, ck, 1.0f), sl2 = fmaf(-cl, cl, 1.0f);
    if (!(sk2 >= 1.0e-5f) || !(sl2 >= 1.0e-5f)) return 0;
    const float rk = rsqrtf(sk2), rl = rsqrtf(sl2);
    float sp, cp;
    sincospif(fmaf(2.0f, u32of(e.x), -1.0f), &sp, &cp);
    const float sk = sk2 * rk, sl = sl2 * rl;
    const float fk[10] = {ck * ck * sl2,
                          0.5f * sk2 * (1.0f - sl2 * cp * cp),
                          0.5f * sk2 * (1.0f - sl2 * sp * sp),
                          sk2 * sl2 * sp * cp,
                          1.41421356f * sk * ck * sl * cl * cp,
                          -1.41421356f * sk * ck * sl * cl * sp,
                          sl2 * (1.0f / 3.0f),
                          0.81649658f * sk * sl * cl * cp,
                          -0.81649658f * sk * sl * cl * sp,
                          1.15470054f * ck * sl2};
    float A = 0.0f;
#pragma unroll
    for (int k = 0; k < 10; ++k) A = fmaf(f.h[k], fk[k], A);
    const float lhs = u32of(e.z) * f.MO;
    const float dl = f.MO * 9.5367431640625e-07f;
    const float band = 6.0f * f.MO * (5.0e-7f * (rk + rl) + 2.0e-6f);
    if (lhs + dl < A - band) return 1;
    if (lhs - dl > A + band) return -1;
    return 0;
}


// The decay-time model (angles = false) and the 4D model.
template <bool ANGLES>
struct TimeGen {
    static constexpr bool kQuickKeeps = !ANGLES, kQuick64 = !ANGLES;
    static constexpr int kBlocksPerSm = 4;
    static constexpr int kUnroll = ANGLES ? 2 : 1;    // two candidates' Philox chains at once
    static constexpr int kBlockEvents = ANGLES ? 0 : 512;
    struct Shared {
        Consts c;
        Filter32 f;
        Exp32 e;
        float near;       // tau above it: z <= -4.3
        float dl;         // bound of the error of u M_T
        double t_lo, span;
        // the test away from the peak on the words themselves (4D): for a first word above
        // far, g = 2^(word lin + con) and the candidate is dropped if its third word > g per_g + more
        uint32_t far;
        float lin, con, per_g, more;
    };

    __device__ static void setup(Shared& S, const GenArgs& A) {
        const double* src = reinterpret_cast<const double*>(A.consts);
        double* dst = reinterpret_cast<double*>(&S.c);
        for (int i = threadIdx.x; i < kConstsDoubles; i += blockDim.x) dst[i] = src[i];
        __syncthreads();
        if (threadIdx.x != 0) return;
        const Consts& c = S.c;
        S.t_lo = A.m.t_lo;
        S.span = __dsub_rn(A.m.t_hi, A.m.t_lo);
        Filter32& f = S.f;
        f.d = (float)(A.m.t_lo - c.mu);
        f.span = (float)S.span;
        f.Gamma = (float)c.Gamma;
        f.c_exp = (float)c.c_exp;
        f.Gs2 = (float)c.Gs2;
        f.k_z = (float)c.k_z;
        f.MT = (float)c.MT;
        f.MO = (float)c.MO;
        for (int k = 0; k < 10; ++k) f.h[k] = (float)c.h[k];
        S.e = exp32_of(c.Gamma, c.c_exp);
        // (a negative sigma has no such region: every candidate takes the full test)
        S.near = c.k_z > 0.0 ? (float)(c.Gs2 + 4.3 / c.k_z) * 1.000001f + 1.0e-6f * (f.span + fabsf(f.d)) : INFINITY;
        S.dl = f.MT * 1.5e-6f;
        // tau = (t_lo - mu) + u span with u = word 2^-32 within 2^-31: the exponent's error is
        // below 2^-24 times 3 |x span| + 2 |con| (the word's, lin's, con's and the sum's roundings),
        // ex2.approx adds 2^-22; a factor 2 and 1e-6 to spare, and 1.5e-6 M_T for u M_T
        const double x = c.Gamma * kLog2e, d = A.m.t_lo - c.mu;
        const double con = c.c_exp * kLog2e - x * d, size = fabs(x) * S.span + fabs(con);
        const double err = 2.0 * (0.7 * 0x1p-22 * size + 2.5e-7) + 1.0e-6;
        const double at = ((double)S.near - d) / S.span;       // u at the end of the peak
        S.far = at < 0.0 ? 0u : (at < 0.999999 ? (uint32_t)((at + 1.0e-6) * 4294967296.0) : 0xFFFFFFFFu);
        if (!(err <= 1.0e-3) || !(c.MT >= 0x1p-90) || !(at < 1.0)) S.far = 0xFFFFFFFFu;   // no such test
        S.lin = (float)(-x * S.span * 0x1p-32);
        S.con = (float)con;
        S.per_g = (float)(4294967296.0 / c.MT * (1.0 + err) * 1.000001);
        S.more = 6500.0f;                                      // 1.5e-6 2^32
    }

    __device__ static bool usable(const Shared& S) {
        const Consts& c = S.c;
        return isfinite(c.MT) && c.MT > 0.0 && isfinite(c.MO) && c.MO > 0.0 && isfinite(c.IT) && c.IT > 0.0;
    }

    // integral of g A over the box (I_T 16 pi / 9) over the envelope's (M_T M_Omega span 8 pi)
    __device__ static void acceptance(const GenArgs& A, float* acc) {
        if (threadIdx.x != 0) return;
        const Consts& c = *A.consts;
        float v = (float)c.IT / ((float)c.MT * (float)(A.m.t_hi - A.m.t_lo));
        if (ANGLES) v *= (2.0f / 9.0f) / (float)c.MO;
        *acc = v;
    }

    // The decay-time test away from the resolution peak, where g is the exponential alone.
    __device__ __forceinline__ static GenCode quick(const Shared& S, const GenArgs& A, const GenIdx& j) {
        const U4 a = gen_draw(A, j, 0u);
        if (ANGLES) {
            const float g = ex2_approx(fmaf(__uint2float_rn(a.x), S.lin, S.con));
            return a.x > S.far && __uint2float_rn(a.z) > fmaf(g, S.per_g, S.more) ? kDrop : kTest32;
        }
        const float tau = fmaf(u32of(a.x), S.f.span, S.f.d);
        const float arg = fmaf(-S.e.x, tau, S.e.off);
        const float g = exp2f(arg);
        const float lhs = u32of(a.z) * S.f.MT;
        const float err = exp32_err(fabsf(S.e.x), fabsf(S.e.off), tau, tau32_err(tau, S.f.d, S.f.span));
        if (!(tau > S.near) || !(fabsf(arg) <= kMaxArg) || !(err <= 1.0e-3f)) return kTest32;
        return decide32(lhs, S.dl, g, g * err);
    }

    __device__ __forceinline__ static GenCode test32(const Shared& S, const GenArgs& A, const GenIdx& j) {
        const U4 a = gen_draw(A, j, 0u);
        int d = time_filter(S.f, a.x, a.z);
        if (d < 0) return kDrop;
        if (!ANGLES) return d > 0 ? kKeep : kTest64;
        const U4 b = gen_draw(A, j, 1u);
        const U4 e = gen_draw(A, j, 2u);
        const int f = angle_filter(S.f, b, e);
        if (f < 0) return kDrop;
        return d > 0 && f > 0 ? kKeep : kTest64;
    }

    __device__ __noinline__ static bool test64(const Shared& S, const GenArgs& A, const GenIdx& j) {
        const U4 a = gen_draw(A, j, 0u);
        const double t = __dadd_rn(S.t_lo, __dmul_rn(u01_int(a.x, a.y), S.span));
        if (!(__dmul_rn(u01_int(a.z, a.w), S.c.MT) < time_pdf(S.c, t))) return false;
        if (!ANGLES) return true;
        const U4 b = gen_draw(A, j, 1u);
        const U4 e = gen_draw(A, j, 2u);
        return __dmul_rn(u01_int(e.z, e.w), S.c.MO) <
               angular_pdf(S.c, sym_int(b.x, b.y), sym_int(b.z, b.w), __dmul_rn(kPi, sym_int(e.x, e.y)));
    }

    __device__ __forceinline__ static void signal(const Shared& S, const GenArgs& A, const GenIdx& j, int64_t pos) {
        const U4 a = gen_draw(A, j, 0u);
        A.t[pos] = __dadd_rn(S.t_lo, __dmul_rn(u01_int(a.x, a.y), S.span));
        if (!ANGLES) return;
        const U4 b = gen_draw(A, j, 1u);
        const U4 e = gen_draw(A, j, 2u);
        A.ck[pos] = sym_int(b.x, b.y);
        A.cl[pos] = sym_int(b.z, b.w);
        A.phi[pos] = __dmul_rn(kPi, sym_int(e.x, e.y));
    }

    // background: uniform in the box, always kept
    __device__ __forceinline__ static void background(const Shared& S, const GenArgs& A, const GenIdx& i, int64_t pos) {
        const U4 a = gen_draw(A, i, 4u);
        A.t[pos] = __dadd_rn(S.t_lo, __dmul_rn(u01_int(a.x, a.y), S.span));
        if (!ANGLES) return;
        const U4 b = gen_draw(A, i, 5u);
        A.ck[pos] = sym_int(a.z, a.w);
        A.cl[pos] = sym_int(b.x, b.y);
        A.phi[pos] = __dmul_rn(kPi, sym_int(b.z, b.w));
    }

    __device__ __forceinline__ static void fill_nan(const GenArgs& A, int64_t pos) {
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        A.t[pos] = nan;
        if (ANGLES) A.ck[pos] = A.cl[pos] = A.phi[pos] = nan;
    }
};

// The tagged model: candidate j of toy k takes (t, u) from call 0 and the tag
// from the first uniform of call 1 (q = +1 if u_q <= 1/2, which is the top bit
// of its first word being clear), and is kept iff u M_S < S(t - mu, q) with S
// in FP64 with the exact forms of tagged.cuh.  Background event i takes t and q
// from call 4.
//
// FP32: away from the peak the four convolutions are exponentials; quick()
// drops a candidate that the oscillation's amplitude cannot lift over its
// threshold (nine in ten) without drawing the tag, test32() evaluates the
// oscillation, near the peak with FP32 erfc and Faddeeva functions.
struct TagGen {
    static constexpr bool kQuickKeeps = false, kQuick64 = false;
    static constexpr int kBlocksPerSm = 3, kUnroll = 1, kBlockEvents = 0;
    struct Shared {
        TagConsts c;
        Conv32 v;
        Phase32 ph;
        float aH, aL, Ds, MS, dl;
        double t_lo, span;
        float f_span;
    };

    __device__ static void setup(Shared& S, const GenArgs& A) {
        const double* src = reinterpret_cast<const double*>(A.consts);
        double* dst = reinterpret_cast<double*>(&S.c);
        for (int i = threadIdx.x; i < kTagConstsDoubles; i += blockDim.x) dst[i] = src[i];
        __syncthreads();
        if (threadIdx.x != 0) return;
        S.t_lo = A.m.t_lo;
        S.span = __dsub_rn(A.m.t_hi, A.m.t_lo);
        S.f_span = (float)S.span;
        S.v = conv32_of(S.c, A.m.t_lo - S.c.mu, S.span);
        S.ph = phase32_of(S.c.Dm, S.c.ph0, A.m.t_lo - S.c.mu, S.span);
        S.aH = (float)S.c.aH;
        S.aL = (float)S.c.aL;
        S.Ds = (float)S.c.Ds;
        S.MS = (float)S.c.MS;
        S.dl = S.MS * 1.5e-6f;
    }

    __device__ static bool usable(const Shared& S) {
        return isfinite(S.c.MS) && S.c.MS > 0.0 && isfinite(S.c.N) && S.c.N > 0.0;
    }

    // N is the integral over both tags, each drawn half of the time
    __device__ static void acceptance(const GenArgs& A, float* acc) {
        if (threadIdx.x != 0) return;
        const TagConsts& c = *reinterpret_cast<const TagConsts*>(A.consts);
        *acc = 0.5f * (float)c.N / ((float)c.MS * (float)(A.m.t_hi - A.m.t_lo));
    }

    __device__ __forceinline__ static GenCode quick(const Shared& S, const GenArgs& A, const GenIdx& j) {
        const U4 a = gen_draw(A, j, 0u);
        const float tau = fmaf(u32of(a.x), S.f_span, S.v.d);
        const float lhs = u32of(a.z) * S.MS;
        const Far32 g = conv32_far(S.v, tau, tau32_err(tau, S.v.d, S.f_span));
        if (!g.ok) return kTest32;
        const float most = S.aH * g.H + S.aL * g.L + fabsf(S.Ds) * g.C;
        return lhs - S.dl > most * (1.0f + g.err) ? kDrop : kTest32;
    }

    __device__ __forceinline__ static GenCode test32(const Shared& S, const GenArgs& A, const GenIdx& j) {
        const U4 a = gen_draw(A, j, 0u);
        const U4 b = gen_draw(A, j, 1u);
        const float tau = fmaf(u32of(a.x), S.f_span, S.v.d);
        const float q = (b.x >> 31) ? -1.0f : 1.0f;
        const Time32 g = conv32(S.v, tau, tau32_err(tau, S.v.d, S.f_span), phase32(S.ph, a.x), S.ph.ok);
        const float sig = S.aH * g.H + S.aL * g.L + q * S.Ds * g.Ci;
        const float err = (S.aH * g.H + S.aL * g.L + fabsf(S.Ds) * g.C) * g.err;
        return decide32(u32of(a.z) * S.MS, S.dl, sig, err);
    }

    __device__ __noinline__ static bool test64(const Shared& S, const GenArgs& A, const GenIdx& j) {
        const U4 a = gen_draw(A, j, 0u);
        const U4 b = gen_draw(A, j, 1u);
        const double t = __dadd_rn(S.t_lo, __dmul_rn(u01_int(a.x, a.y), S.span));
        return __dmul_rn(u01_int(a.z, a.w), S.c.MS) < tag_signal(S.c, t, tag_of(b.x));
    }

    __device__ __forceinline__ static double tag_of(uint32_t hi) { return (hi >> 31) ? -1.0 : 1.0; }

    __device__ __forceinline__ static void signal(const Shared& S, const GenArgs& A, const GenIdx& j, int64_t pos) {
        const U4 a = gen_draw(A, j, 0u);
        const U4 b = gen_draw(A, j, 1u);
        A.t[pos] = __dadd_rn(S.t_lo, __dmul_rn(u01_int(a.x, a.y), S.span));
        A.q[pos] = tag_of(b.x);
    }

    __device__ __forceinline__ static void background(const Shared& S, const GenArgs& A, const GenIdx& i, int64_t pos) {
        const U4 a = gen_draw(A, i, 4u);
        A.t[pos] = __dadd_rn(S.t_lo, __dmul_rn(u01_int(a.x, a.y), S.span));
        A.q[pos] = tag_of(a.z);
    }

    __device__ __forceinline__ static void fill_nan(const GenArgs& A, int64_t pos) {
        A.t[pos] = A.q[pos] = __longlong_as_double(0x7ff8000000000000ll);
    }
};

}  // namespace
}  // namespace ipa

extern "C" ipa_status ipa_toygen(const ipa_model* model, const double* theta_dev, uint64_t seed,
                                 int32_t n_toys, const int64_t* n_sig_dev, const int64_t* n_bkg_dev,
                                 const int64_t* offsets_dev, const ipa_event_buffers* out,
                                 void* stream) {
    using namespace ipa;
    ipa_status st = check_model(model);
    if (st != IPA_OK) return st;
    if (n_toys < 0 || !out || !theta_dev) {
        set_error("ipa_toygen: bad arguments");
        return IPA_ERR_ARG;
    }
    if (n_toys == 0) return IPA_OK;
    if (!n_sig_dev || !n_bkg_dev || !offsets_dev || !out->t || out->capacity < 0) {
        set_error("ipa_toygen: NULL count, offset or output column");
        return IPA_ERR_ARG;
    }
    const bool four = model->kind == IPA_MODEL_ANGTIME4D;
    if (four && (!out->ck || !out->cl || !out->phi)) {
        set_error("ipa_toygen: the 4D model needs ck, cl and phi output columns");
        return IPA_ERR_ARG;
    }
    const bool phis = model->kind == IPA_MODEL_PHIS;
    if (phis && (!out->ck || !out->cl || !out->phi || !out->q)) {
        set_error("ipa_toygen: the phi_s model needs ck, cl, phi and q output columns");
        return IPA_ERR_ARG;
    }
    const bool tag = model->kind == IPA_MODEL_TAGGED1D;
    if (tag && !out->q) {
        set_error("ipa_toygen: the tagged model needs a q output column");
        return IPA_ERR_ARG;
    }
    Scratch* sc = nullptr;
    if ((st = scratch_get(1, 2, &sc)) != IPA_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const ModelDev m{model->kind, model->n_par, model->t_lo, model->t_hi};
    if ((st = launch_consts(m, theta_dev, 1, sc->consts, s)) != IPA_OK) return st;
    GenArgs a{};
    a.m = m;
    a.consts = sc->consts;
    a.keys = PhiloxKeys(seed);
    a.n_toys = n_toys;
    a.n_sig = n_sig_dev;
    a.n_bkg = n_bkg_dev;
    a.offsets = offsets_dev;
    a.capacity = out->capacity;
    a.t = out->t;
    a.ck = out->ck;
    a.cl = out->cl;
    a.phi = out->phi;
    a.q = out->q;
    if (tag) return launch_generator<TagGen>(a, s);
    if (phis) return launch_phis_toygen(a, s);
    if (four) return launch_generator<TimeGen<true>>(a, s);
    return launch_generator<TimeGen<false>>(a, s);
}
