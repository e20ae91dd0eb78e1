// Hot-path steps a2-a6: per-event normalised PDF, -w log P, fused analytic
// adjoint and the deterministic FP64 reduction, for one fit or for many
// segments (fits) packed back to back.
//
// Sec. 3 of the paper evaluates the PDF with one thread per event, takes the
// log of the signal/background mixture in a second launch and sums the logs
// on the host.  Here one kernel does all of it.  Work is split into 512-event
// tiles owned by single warps: lane l accumulates events l, l+32, ..., l+480
// of its tile in order (coalesced 8-byte loads), the warp reduces its FP64
// accumulators with a fixed butterfly and writes one partial per tile.
// The warp that completes the last tile of a group of 32 tiles reduces the
// group, and the warp that completes a segment's last group adds its group
// partials in fixed order and writes the NLL and gradient.  No block-wide
// barrier sits in the event loop, and the result does not depend on the
// launch geometry (block size, grid, tiles taken at once).
//
// The GPU has 2 FP64 operations per clock per SM, so the per-event arithmetic
// is arranged to spend as few of them as possible:
//   * the decay-time term uses erfc(z) = 2 - exp(-z^2) erfcx(|z|) for z < 0 and
//     erfc(z) = exp(-z^2) erfcx(z) for z >= 0, with exp(-Gamma tau + Gamma^2
//     sigma^2/2) exp(-z^2) = exp(-tau^2/(2 sigma^2)): the Gaussian factor that
//     the gradient needs anyway replaces the exponential inside erfc;
//   * sin/cos, the whole angular basis, A and the ten angular sums, the decay
//     exponential, the Gaussian and erfcx run on the integer pipe in 64-bit
//     fixed point at four to six instructions per product (fast_fixed.cuh); the
//     rows that allow it (Angtime, Time1d below) leave about 15 FP64 instructions per event;
//   * sin(theta_K) sin(theta_mu) is one square root; the constant factors of
//     the ten angular functions are folded into the amplitude coefficients.
//
// Gradient (fused adjoint).  With r = w/P, every derivative of the NLL is a
// contraction of a few per-event sums with parameter-only factors:
//   S_k = sum r T f_k,  D_j = sum r A dT/dtheta_j (j = Gamma, sigma, mu),
//   Q = sum r,          SH = sum_k h_k S_k = sum r T A,
//   dNLL/dtime_j = -cs D_j + cs (dI_T/dtheta_j / I_T) SH,
//   dNLL/df_b    = SH / (I_T I_Omega) - Q / V,
//   dNLL/dang_j  = -cs sum_k (dh_k/dtheta_j) S_k,   cs = (1 - f_b)/(I_T I_Omega),
// so the event pass carries 15 accumulators (4D) instead of one per
// parameter and the angular derivatives cost nothing per event.
#include <math.h>

#include <type_traits>

#include "fp64_math.cuh"
#include "int_math.cuh"
#include "angular.cuh"
#include "fast_fixed.cuh"
#include "ipa_internal.cuh"
#include "team_tile.cuh"
#include "tile_reduce.cuh"

namespace ipa {
namespace {

constexpr int kNllBlock = 128;                       // threads per block of the basis kernel

// A warp keeps a copy of its segment's record (Consts, with the factors the event
// loop multiplies by in its part k: NllCoef) in shared memory.

// The part of the decay-time factor that needs the Gaussian and erfcx, for an
// event with t <= tcut (z >= -6.25 up to rounding): with g = exp(-tau^2 /
// (2 sigma^2)) and X = erfcx(|z|), returns g X in .x and g in .y, the sign of
// .y carrying z >= 0 (negative) or z < 0 (positive).  Then 2 g(tau) = 2E - gX
// (z < 0) or gX (z >= 0).  Events with t > tcut have 2 g(tau) = 2E to 1e-17
// relative and a Gaussian below 1e-17; they are given (0, +0).
__device__ __forceinline__ double2 gauss_erfcx(const Consts& c, double tau, const MathTables* mt) {
    // branch-free integer exp; the argument is clamped at -705 (events more
    // than 37 sigma before mu), where the Gaussian, below 1e-306, is nothing
    // against the exponential term of 2 g(tau)
    const double gr = -(tau * tau) * c.k_g;
    const double g = fx_exp_neg(below_neg(gr, -705.0) ? -705.0 : gr, mt);
    const double z = (c.Gs2 - tau) * c.k_z;
    const double x = fabs(z);
    const bool zneg = negative(z);
    double X = fx_erfcx(x, mt);
    if (above(x, 6.25)) {
        // z < 0: the erfcx term is below 1e-17 of E; z >= 0 (tau far below the
        // resolution peak, outside the usual range): exact library erfcx
        X = zneg ? 0.0 : erfcx(x);
    }
    return make_double2(g * X, zneg ? g : -g);
}

// A' = sum_k hq_k f_k in FP64 (cached basis, or angles outside fx_angles_ok).
__device__ __forceinline__ double amplitude_sum(const double* hq, const double* f) {
    double Ap = hq[0] * f[0];
#pragma unroll
    for (int k = 1; k < 10; ++k) Ap = fma(hq[k], f[k], Ap);
    return Ap;
}

// One event: the log term (w log P added to acc[0], or for w = 1 exactly, P
// folded into the lane's product) and the adjoint sums.  For the 4D model f
// holds either the unscaled products f'_k (CACHED = false) or the cached basis
// f_k (CACHED = true); Ap = (cs/2) A (c.k.aq for the 1D model); ge is the
// event's gauss_erfcx value or (0, +0).
// Accumulators (kD = 12 for 4D, 3 for 1D), with r = w / P and A' = (cs/2) A:
//   acc[1] = sum r,  acc[2 + k] = sum r T2 f_k (4D) or acc[2] = sum r T2 (1D),
//   acc[kD] = sum r A' tau T2,  acc[kD + 1] = sum r A' Gx,  acc[kD + 2] = sum r A' tau Gx;
// the derivatives in Gamma, sigma and mu are linear in these (finalize).
template <int KIND, bool GRAD, bool CACHED, bool WEIGHTED>
__device__ __forceinline__ void event(const Consts& c, const MathTables* mt, double t, const double* f,
                                      double Ap, double w, double2 ge, double* acc, double* prod, int* esum) {
    const double tau = t - c.mu;
    const double E2 = exp_int(fma(-c.Gamma, tau, c.k.c2), mt);
    const long long gb = __double_as_longlong(ge.y);
    const double T2 = gb >= 0 ? E2 - ge.x : ge.x;
    const double Gx = __longlong_as_double(gb & 0x7FFFFFFFFFFFFFFFll);
    const double P = fma(T2, Ap, c.cb);
    // events of weight exactly 1 (all events without a weight column) join the
    // lane's log product, so a column of ones gives the same bits as no column
    if (WEIGHTED && __double_as_longlong(w) != 0x3FF0000000000000ll)
        acc[0] = fma(w, log_fast(P, mt), acc[0]);
    else
        log_mul(P, prod, esum);
    if (GRAD) {
        // r = w / P feeds only the adjoint sums; its ~6e-14 relative error
        // (rcp_newton) is far inside the gradient's tolerance
        const double r = WEIGHTED ? w * rcp_newton(P) : rcp_newton(P);
        acc[1] += r;
        const double rT = r * T2;
        constexpr int kD = KIND == IPA_MODEL_ANGTIME4D ? 12 : 3;
        if (KIND == IPA_MODEL_ANGTIME4D) {
#pragma unroll
            for (int k = 0; k < 10; ++k) acc[2 + k] = fma(rT, f[k], acc[2 + k]);
        } else {
            acc[2] += rT;
        }
        const double rA = r * Ap;
        const double u = rA * tau;
        acc[kD + 0] = fma(u, T2, acc[kD + 0]);
        acc[kD + 1] = fma(rA, Gx, acc[kD + 1]);
        acc[kD + 2] = fma(u, Gx, acc[kD + 2]);
    }
}

// Write NLL (and gradient) of one segment from its reduced accumulators.
// With S_k = sum r T f_k and SH = sum_k h_k S_k = sum r T A (A = 1 in 1D), and
// D_j = sum r A dT/dtheta_j where
//   dT/dGamma = (Gamma sigma^2 - tau) T - sigma^2 G,
//   dT/dsigma = Gamma^2 sigma T - (tau / sigma + Gamma sigma) G,
//   dT/dmu    = Gamma T - G,   G = cG Gx,
// the accumulators give cs D_Gamma = cs Gamma sigma^2 SH - Y1 - 2 sigma^2 cG Y2,
// cs D_sigma = cs Gamma^2 sigma SH - 2 cG (Y3 / sigma + Gamma sigma Y2) and
// cs D_mu = cs Gamma SH - 2 cG Y2 (Y1..Y3 = acc[kD..kD+2]).
template <int KIND, bool GRAD, bool CACHED>
__device__ void finalize(const Consts& c, const double* acc, int n_par, double* out, int lane) {
    // every lane holds acc; lane j writes component j (0: the NLL, 1 + j: the
    // derivative in parameter j), computing only what that component needs
    if (lane == 0) out[0] = -acc[0];
    if (!GRAD) return;
    const double Q = acc[1];
    constexpr int kD = KIND == IPA_MODEL_ANGTIME4D ? 12 : 3;
    double S[10];
    double SH;
    if (KIND == IPA_MODEL_ANGTIME4D) {
        SH = 0.0;
        for (int k = 0; k < 10; ++k) {
            S[k] = (CACHED ? 0.5 : 0.5 * kBasisScale[k]) * acc[2 + k];
            SH = fma(c.h[k], S[k], SH);
        }
    } else {
        SH = 0.5 * acc[2];
    }
    const double csSH = c.cs * SH;
    const double Y1 = acc[kD], Y2 = acc[kD + 1], Y3 = acc[kD + 2];
    const double tcG = 2.0 * c.cG;
    if (lane < 3) {
        double csD;
        if (lane == 0) csD = fma(c.Gs2, csSH, -fma(tcG * c.s2, Y2, Y1));
        else if (lane == 1) csD = fma(c.G2s, csSH, -tcG * fma(c.inv_s, Y3, c.Gsig * Y2));
        else csD = fma(c.Gamma, csSH, -tcG * Y2);
        out[1 + lane] = fma(c.dlnIT[lane], csSH, -csD);
    } else if (lane == IPA_FB) {
        out[1 + IPA_FB] = fma(SH, c.inv_ITIO, -Q * c.inv_V);
    } else if (KIND == IPA_MODEL_ANGTIME4D && lane < IPA_NPAR_4D) {
        const int j = lane - IPA_A0SQ;
        double s = 0.0;
        for (int k = 0; k < 10; ++k) s = fma(c.dh[k][j], S[k], s);
        out[1 + lane] = -c.cs * s;
    }
    for (int j = (KIND == IPA_MODEL_ANGTIME4D ? IPA_NPAR_4D : IPA_NPAR_1D) + lane; j < n_par; j += 32)
        out[1 + j] = 0.0;
}

// The plain loop over rows [i0, i1) of a tile, events below ev1: lane l adds events l, l + 32,
// ... in order into acc (and the log product).
template <int KIND, bool GRAD, bool CACHED, bool WEIGHTED>
__device__ __forceinline__ void plain_rows(const Consts& c, const MathTables* mt, const Cols& cols, int i0, int i1,
                                           int64_t tbase, int64_t ev1, double2* sbuf, int lane, double* acc,
                                           double* prod, int* esum) {
    const unsigned below = (1u << lane) - 1u;
#pragma unroll 1
    for (; i0 < i1; i0 += kSub) {
        SlowRows r;
        slow_rows(r, cols, c.k.tcut, tbase, i0, ev1, sbuf, lane,
                  [&](int64_t e) { return gauss_erfcx(c, __ldg(cols.t + e) - c.mu, mt); });
#pragma unroll 1
        for (int q = 0; q < kSub; ++q) {
            const int64_t e = tbase + lane + 32 * (i0 + q);
            if (e < ev1) {
                const int j = r.at(q, below, lane);
                const double2 ge = j >= 0 ? sbuf[j] : make_double2(0.0, 0.0);
                const double w = WEIGHTED ? __ldg(cols.w + e) : 1.0;
                double f[10];
                double Ap = c.k.aq;
                if (KIND == IPA_MODEL_ANGTIME4D) {
                    if (CACHED) {
#pragma unroll
                        for (int k = 0; k < 10; ++k) f[k] = __ldg(cols.fk + k * cols.fk_stride + e);
                        Ap = amplitude_sum(c.k.hc, f);
                    } else {
                        const double ck = __ldg(cols.ck + e), cl = __ldg(cols.cl + e), phi = __ldg(cols.phi + e);
                        if (c.k.fixed && fx_angles_ok(ck, cl, phi)) {
                            // the angular products and A on the integer pipe
                            long long g[10];
                            fx_basis(ck, cl, phi, mt, g);
                            long long A = 0;
#pragma unroll
                            for (int k = 0; k < 10; ++k) A = fx_mad(Fx{c.k.ga[k].x, c.k.ga[k].y}, fx(g[k]), A);
                            Ap = fx_to_double(A, c.k.hexp);
                            const long long F[10] = {g[0] - g[2], g[1] - g[3], g[1] - g[2] + g[3], g[4], g[5],
                                                     g[6], g[0], g[7], g[8], g[9]};
#pragma unroll
                            for (int k = 0; k < 10; ++k) f[k] = fx_to_double(F[k], 0);
                        } else {
                            basis_unscaled(ck, cl, phi, mt, f);
                            Ap = amplitude_sum(c.k.hq, f);
                        }
                    }
                }
                event<KIND, GRAD, CACHED, WEIGHTED>(c, mt, __ldg(cols.t + e), f, Ap, w, ge, acc, prod,
                                                    esum);
            }
        }
        __syncwarp();
    }
}

// ---- the fixed-point path of NLL + gradient ----
// On this GPU a warp FP64 instruction occupies the sub-partition's FP64 unit
// for about 64 cycles (2 FP64 operations per clock per SM), so everything with
// a known range runs in 64-bit fixed point (fast_fixed.cuh): the decay
// exponential, the angular basis, A', the ten angular sums and the 1D model's sums.
// What stays FP64: P, 1/P, the log (or the product of the P's), and for the 4D model the
// four sums with r, tau and the Gaussian.
//
// The angular sums: r T is converted once per event to signed fixed point, in units of
// 2^(top - 63), each product with a basis function (Q62) is the high part of the
// 128-bit product (units of 2^(top - 61)), and a lane adds its events exactly in
// 64-bit integers and converts each sum to a double once per tile (sums of f'_k
// are differences of sums of basis functions, taken in integers).  top follows
// the segment's typical r T (NllCoef::rtop) and the largest weight of the tile,
// so a unit is 2^-48 of a typical term; error of a sum: 0.41 units rms per
// event, of random sign, below that of the reciprocal r (6e-14 relative).  The 1D
// model: sums of r T and r Gx and their products with tau, as in the tagged model
// (tagged.cu).  Lanes outside the ranges are fixed up in FP64.  A tile in which some P lies outside the Newton reciprocal's range (zero,
// subnormal, negative, huge, infinite or NaN) or some |r T| >= 2^(top - 3) is redone
// by the plain loop.  Either way the tile's sums depend only on its events, never
// on the launch geometry (team_tile.cuh).
//
// The cached basis takes the same path (its f_k converted to Q62, |f_k| < 1.5): 4.2e6 events
// 327 us by the plain loop, 239 here, weighted 431 and 267; 1000 events 58 and 32 (teams).
//
// Measured (one pass of the public call, 512 toys of 20 000 events, then 1e7
// weighted events): the angular products, A and the exponential in FP64 and
// 14-instruction 64-bit products, an FP64 multiply-add per angular sum: 1060 and
// 1073 us; this path: 643 and 685 (now 608, with the records by block, and 689).
// About 1060 warp instructions per row occupy the FP64 unit 60 %, the two 32-bit
// multiplier and adder pipes 50 % each and the issue slots 50 %; 128 registers
// leave 16 warps per SM, and launch bounds for 20 or 24 cost more in spills than
// they hide (728 and 760 us).

// The integer-pipe results of one event that its FP64 work needs.
struct RowIn {
    double tau, w, E2, Ap;
    Fx g[10];   // fx_basis, or the cached basis
};

// The FP64 values for a lane outside the fixed-point ranges (rare): the basis, A'
// (with the f'_k in the plain loop's order) and the exponential.  Basis values beyond
// the fixed-point range (|cos| > 1, angles that are NaN or infinite) make A' a NaN, so
// that the tile is redone by the plain loop.
__device__ __noinline__ void fix_row(const Consts& c, const MathTables* mt, double t, double ck, double cl, double phi,
                                     bool ok_exp, RowIn& v) {
    if (!ok_exp) v.E2 = exp_fast(fma(-c.Gamma, v.tau, c.k.c2), mt);
    if (!fx_angles_ok(ck, cl, phi)) {
        double f[10];
        basis_unscaled(ck, cl, phi, mt, f);
        v.Ap = amplitude_sum(c.k.hq, f);
        const double sk2 = fma(-ck, ck, 1.0), G = sk2 * f[6], gcc = sk2 - f[1];
        const double g[10] = {f[6], sk2, G, gcc, f[3], f[4], f[5], f[7], f[8], f[9]};
#pragma unroll
        for (int k = 0; k < 10; ++k) {
            if (!fits_q62(g[k])) v.Ap = __longlong_as_double(0x7ff8000000000000ll);
            v.g[k] = fx(to_q62_nb(g[k]));
        }
    }
}

// (the same register-saving detour for the exponential)
__device__ __noinline__ double fix_exp(const Consts& c, const MathTables* mt, double tau) {
    return exp_fast(fma(-c.Gamma, tau, c.k.c2), mt);
}

// (and the largest |f_k| of the cached basis, by its high word)
__device__ __forceinline__ void load_cached_row(const Consts& c, const MathTables* mt, const Cols& cols, int64_t e,
                                                RowIn& v, int* f_most) {
    const double t = __ldg(cols.t + e);
    v.tau = t - c.mu;
    long long A = 0;
#pragma unroll
    for (int k = 0; k < 10; ++k) {
        const double f = __ldg(cols.fk + k * cols.fk_stride + e);
        *f_most = max(*f_most, high_word(f));
        v.g[k] = fx(fx_signed(f, 1));
        A = fx_mad(Fx{c.k.gc[k].x, c.k.gc[k].y}, v.g[k], A);
    }
    v.Ap = fx_to_double(A, c.k.cexp);
    bool ok = fx_in_range(t, c.k.ex.top);
    v.E2 = fx_exp(fx(fx_signed(t, c.k.ex.top)), c.k.ex, mt, &ok);
    if (!ok) v.E2 = fix_exp(c, mt, v.tau);
}

__device__ __forceinline__ void load_row(const Consts& c, const MathTables* mt, const Cols& cols, int64_t e, RowIn& v) {
    const double t = __ldg(cols.t + e);
    const double ck = __ldg(cols.ck + e), cl = __ldg(cols.cl + e), phi = __ldg(cols.phi + e);
    v.tau = t - c.mu;
    bool ok_exp = fx_in_range(t, c.k.ex.top);
    v.E2 = fx_exp(fx(fx_signed(t, c.k.ex.top)), c.k.ex, mt, &ok_exp);
    long long g[10];
    fx_basis(ck, cl, phi, mt, g);
    long long A = 0;
#pragma unroll
    for (int k = 0; k < 10; ++k) {
        v.g[k] = fx(g[k]);
        A = fx_mad(Fx{c.k.ga[k].x, c.k.ga[k].y}, v.g[k], A);
    }
    v.Ap = fx_to_double(A, c.k.hexp);
    if (__any_sync(__activemask(), !(ok_exp && fx_angles_ok(ck, cl, phi)))) {
        RowIn x = v;                         // (a copy, so that v itself stays in registers)
        fix_row(c, mt, t, ck, cl, phi, ok_exp, x);
        v = x;
    }
}

// The models of team_tile.cuh.
template <bool CACHED>
struct Angtime {
    using Record = Consts;
    using Slow = double2;
    // FP64: sum r, sum r A' tau T2, sum r A' Gx, sum r A' tau Gx, sum w log P; integers: r T g_k
    static constexpr int kTopRange = 900, kLeast = 16, kPlainBelow = kFewEvents;
    static constexpr int kSums = 5, kInts = 10, NA = n_acc(IPA_MODEL_ANGTIME4D, true);
    using Sums = FastSums<kSums, kInts>;

    static __device__ __forceinline__ bool usable(const Consts& c, int64_t events, FastScale* sc) {
        sc->top = c.k.rtop;
        sc->gtop = 0;
        return (CACHED ? c.k.cached : c.k.fixed) && events >= kFewEvents;
    }
    template <bool W>
    static __device__ __forceinline__ void quarter(const Consts& c, const MathTables* mt, const Cols& cols, int64_t tbase,
                                                   int i0, int64_t ev1, double2* sbuf, double* wbuf, int lane,
                                                   FastScale sc, Sums& s) {
        const unsigned below = (1u << lane) - 1u;
        SlowRows r;
        slow_rows(r, cols, c.k.tcut, tbase, i0, ev1, sbuf, lane,
                  [&](int64_t e) { return gauss_erfcx(c, __ldg(cols.t + e) - c.mu, mt); });
#pragma unroll 1
        for (int q = 0; q < kSub; ++q) {
            const int64_t e = tbase + lane + 32 * (i0 + q);
            if (e < ev1) {
                const int j = r.at(q, below, lane);
                const double2 ge = j >= 0 ? sbuf[j] : make_double2(0.0, 0.0);
                RowIn v;
                if (CACHED) load_cached_row(c, mt, cols, e, v, &s.tau_most);
                else load_row(c, mt, cols, e, v);
                v.w = W ? wbuf[q * 32 + lane] : 1.0;
                const long long gb = __double_as_longlong(ge.y);
                const double T2 = gb >= 0 ? v.E2 - ge.x : ge.x;
                const double Gx = __longlong_as_double(gb & 0x7FFFFFFFFFFFFFFFll);
                const double P = fma(T2, v.Ap, c.cb);
                add_log<W>(P, v.w, mt, &s.f[4], s);
                const double rr = W ? v.w * rcp_newton_nb(P) : rcp_newton_nb(P);
                s.f[0] += rr;
                const double rT = rr * T2;
                s.most = max(s.most, high_word(rT));
                const long long rq = fx_odd(rT, W ? sc.top : c.k.rtop);
                const int one = rq != 0;
                const Fx R = fx(rq);
#pragma unroll
                for (int k = 0; k < 10; ++k) s.g[k] = fx_mad1(R, v.g[k], s.g[k], one);
                const double rA = rr * v.Ap;
                const double u = rA * v.tau;
                s.f[1] = fma(u, T2, s.f[1]);
                s.f[2] = fma(rA, Gx, s.f[2]);
                s.f[3] = fma(u, Gx, s.f[3]);
            }
        }
        __syncwarp();
    }
    static __device__ __forceinline__ bool bad(const Consts&, FastScale sc, const Sums& s) {
        return p_out_of_range(s) || (s.most >> 20) > 1023 - 4 + sc.top ||
               (CACHED && s.tau_most >= 0x3FF80000);      // |f_k| < 1.5 (coef_scale_cached)
    }
    static __device__ __forceinline__ void accumulators(const Consts&, FastScale sc, const Sums& s, double* acc) {
        const long long S[10] = {s.g[0] - s.g[2], s.g[1] - s.g[3], s.g[1] - s.g[2] + s.g[3], s.g[4], s.g[5],
                                 s.g[6], s.g[0], s.g[7], s.g[8], s.g[9]};
        if (CACHED) {
#pragma unroll
            for (int k = 0; k < 10; ++k) acc[2 + k] = fx_to_double(s.g[k], sc.top + 1);
        }
        acc[0] = s.f[4];
        acc[1] = s.f[0];
#pragma unroll
        for (int k = 0; k < 10; ++k)
            if (!CACHED) acc[2 + k] = fx_to_double(S[k], sc.top + 1);
        acc[12] = s.f[1];
        acc[13] = s.f[2];
        acc[14] = s.f[3];
    }
    template <bool W>
    static __device__ __forceinline__ void plain(const Consts& c, const MathTables* mt, const Cols& cols, int i0, int i1,
                                                 int64_t tbase, int64_t ev1, double2* sbuf, int lane, double* acc,
                                                 double* prod, int* esum) {
        plain_rows<IPA_MODEL_ANGTIME4D, true, CACHED, W>(c, mt, cols, i0, i1, tbase, ev1, sbuf, lane, acc, prod, esum);
    }
    static __device__ __forceinline__ void finish(const Consts& c, const double* acc, int n_par, double* out, int lane) {
        finalize<IPA_MODEL_ANGTIME4D, true, CACHED>(c, acc, n_par, out, lane);
    }
};

struct Time1d {
    using Record = Consts;
    using Slow = double2;
    // FP64: sum r, sum w log P; integers: r T, r Gx, r tau T, r tau Gx (the factor A' = cs/2 outside)
    static constexpr int kTopRange = 400, kLeast = 14, kPlainBelow = 0;
    static constexpr int kSums = 2, kInts = 4, NA = n_acc(IPA_MODEL_TIME1D, true);
    using Sums = FastSums<kSums, kInts>;

    static __device__ __forceinline__ bool usable(const Consts& c, int64_t events, FastScale* sc) {
        // a typical r T is near 1 / max(cs / 2, cb / 2); the Gaussian's tau is taken within 14 to 28 sigma:
        // r Gx is above the sums' unit within 8.6 sigma only, except where P itself falls with the
        // Gaussian (bad)
        sc->top = 10 + 1023 - max(exponent_field(c.k.aq), exponent_field(c.cb) - 1);
        sc->gtop = exponent_field(c.sigma) - 1023 + 5;
        return c.k.ex.ok && sc->gtop >= -400 && sc->gtop <= 400;
    }
    template <bool W>
    static __device__ __forceinline__ void quarter(const Consts& c, const MathTables* mt, const Cols& cols, int64_t tbase,
                                                   int i0, int64_t ev1, double2* sbuf, double* wbuf, int lane,
                                                   FastScale sc, Sums& s) {
        const unsigned below = (1u << lane) - 1u;
        SlowRows r;
        slow_rows(r, cols, c.k.tcut, tbase, i0, ev1, sbuf, lane,
                  [&](int64_t e) { return gauss_erfcx(c, __ldg(cols.t + e) - c.mu, mt); });
#pragma unroll 1
        for (int q = 0; q < kSub; ++q) {
            const int64_t e = tbase + lane + 32 * (i0 + q);
            if (e < ev1) {
                const int j = r.at(q, below, lane);
                const double2 ge = j >= 0 ? sbuf[j] : make_double2(0.0, 0.0);
                const double t = __ldg(cols.t + e), w = W ? wbuf[q * 32 + lane] : 1.0;
                const double tau = t - c.mu;
                bool ok = fx_in_range(t, c.k.ex.top);
                double E2 = fx_exp(fx(fx_signed(t, c.k.ex.top)), c.k.ex, mt, &ok);
                if (!ok) E2 = fix_exp(c, mt, tau);
                const long long gb = __double_as_longlong(ge.y);
                const double T2 = gb >= 0 ? E2 - ge.x : ge.x;
                const double Gx = __longlong_as_double(gb & 0x7FFFFFFFFFFFFFFFll);
                const double P = fma(T2, c.k.aq, c.cb);
                add_log<W>(P, w, mt, &s.f[1], s);
                const double rr = W ? w * rcp_newton_nb(P) : rcp_newton_nb(P);
                s.f[0] += rr;
                const double x[2] = {rr * T2, rr * Gx};
                s.tau_most = max(s.tau_most, high_word(tau));
                const Fx T[2] = {fx(fx_signed(tau, c.k.ex.top)), fx(fx_signed(tau, sc.gtop))};
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    s.most = max(s.most, high_word(x[i]));
                    const long long a = fx_odd(x[i], sc.top);
                    s.g[i] += a;
                    s.g[2 + i] = fx_mad1(fx((long long)((unsigned long long)a << 3)), T[i], s.g[2 + i], a != 0);
                    if (i == 1) s.gtau_most = max(s.gtau_most, a != 0 ? high_word(tau) : 0);
                }
            }
        }
        __syncwarp();
    }
    static __device__ __forceinline__ bool bad(const Consts& c, FastScale sc, const Sums& s) {
        return p_out_of_range(s) || beyond_factor(s.most, sc.top) || beyond_tau(s.tau_most, c.k.ex.top) ||
               beyond_tau(s.gtau_most, sc.gtop);
    }
    static __device__ __forceinline__ void accumulators(const Consts& c, FastScale sc, const Sums& s, double* acc) {
        acc[0] = s.f[1];
        acc[1] = s.f[0];
        acc[2] = fx_to_double(s.g[0], sc.top - 1);
        acc[3] = c.k.aq * fx_to_double(s.g[2], sc.top + c.k.ex.top - 3);
        acc[4] = c.k.aq * fx_to_double(s.g[1], sc.top - 1);
        acc[5] = c.k.aq * fx_to_double(s.g[3], sc.top + sc.gtop - 3);
    }
    template <bool W>
    static __device__ __forceinline__ void plain(const Consts& c, const MathTables* mt, const Cols& cols, int i0, int i1,
                                                 int64_t tbase, int64_t ev1, double2* sbuf, int lane, double* acc,
                                                 double* prod, int* esum) {
        plain_rows<IPA_MODEL_TIME1D, true, false, W>(c, mt, cols, i0, i1, tbase, ev1, sbuf, lane, acc, prod, esum);
    }
    static __device__ __forceinline__ void finish(const Consts& c, const double* acc, int n_par, double* out, int lane) {
        finalize<IPA_MODEL_TIME1D, true, false>(c, acc, n_par, out, lane);
    }
};

template <int KIND, bool CACHED>
using Model = std::conditional_t<KIND == IPA_MODEL_TIME1D, Time1d, Angtime<CACHED>>;

// A segment's record into the warp's copy in shared memory (warp-collective).
__device__ __forceinline__ void load_warp_consts(Consts& c, const Consts* src_consts, int lane) {
    __syncwarp();
    const double* src = reinterpret_cast<const double*>(src_consts);
    double* dst = reinterpret_cast<double*>(&c);
#pragma unroll
    for (int i = lane; i < kConstsDoubles; i += 32) dst[i] = __ldg(src + i);
    __syncwarp();
}

// Blocks of any whole number of warps (1..kMaxWarps); each warp keeps a copy of
// its current segment's constants in dynamic shared memory.
constexpr int kMaxWarps = 8;

template <int KIND, bool GRAD, bool CACHED, bool WEIGHTED>
__global__ void __launch_bounds__(32 * kMaxWarps, 2)
nll_kernel(Cols cols, int64_t n, const int64_t* __restrict__ seg_begin,
           const int64_t* __restrict__ seg_end, const int64_t* __restrict__ seg_tiles, int n_seg,
           const Consts* __restrict__ consts,
           double* __restrict__ partials, unsigned* __restrict__ counters, unsigned* __restrict__ gcount,
           unsigned* __restrict__ work, double* __restrict__ out, int n_par, int per_take) {
    constexpr int NA = n_acc(KIND, GRAD);
    const int out_stride = GRAD ? 1 + n_par : 1;
    __shared__ MathTables mt;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int n_wib = blockDim.x >> 5;
    double2* const sbuf = reinterpret_cast<double2*>(dyn_smem) + wib * (kSub * 32);
    Consts& wc = reinterpret_cast<Consts*>(dyn_smem + (size_t)n_wib * kSub * 32 * sizeof(double2))[wib];
    double* const wbuf = reinterpret_cast<double*>(dyn_smem + (size_t)n_wib * (kSub * 32 * sizeof(double2) + sizeof(Consts))) +
                         wib * (kSub * 32);      // with weights and gradient only

    load_math_tables(&mt);
    __syncthreads();
    // Launched as a programmatic dependent of the constants kernel: the table
    // load above overlaps it; everything below waits for its results.
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const bool single = seg_begin == nullptr;
    const int64_t total = single ? (n + kTile - 1) / kTile : __ldg(seg_tiles + n_seg);

    // empty segments have no tile to finalise them: block 0 writes their zeros
    if (blockIdx.x == 0) {
        for (int s = threadIdx.x; s < n_seg; s += blockDim.x) {
            const bool empty = single ? (n == 0) : (__ldg(seg_tiles + s + 1) == __ldg(seg_tiles + s));
            if (empty) {
                for (int j = 0; j < out_stride; ++j) out[(size_t)s * out_stride + j] = 0.0;
            }
        }
    }

    // Tiles are handed out dynamically, `per_take` consecutive tiles at a time
    // (work[0] counts the takes), so SMs whose warps finish early take more; a
    // tile's partial does not depend on which warp computes it.  The last warp
    // to leave resets both work counters.
    int cur = -1;
    while (true) {
        unsigned taken = 0;
        if (lane == 0) taken = atomicAdd(work, 1u);
        const int64_t first = (int64_t)__shfl_sync(0xffffffffu, taken, 0) * per_take;
        if (first >= total) break;
        const int64_t stop = first + per_take < total ? first + per_take : total;
        for (int64_t tile = first; tile < stop; ++tile) {
            int seg = 0;
            int64_t t0 = 0, t1 = total, ev0 = 0, ev1 = n;
            if (!single) {
                seg = find_segment(seg_tiles, n_seg, tile);
                t0 = __ldg(seg_tiles + seg);
                t1 = __ldg(seg_tiles + seg + 1);
                ev0 = clamp_off(__ldg(seg_begin + seg), n);
                ev1 = clamp_off(__ldg(seg_end + seg), n);
                if (ev1 < ev0) ev1 = ev0;
            }
            if (seg != cur) {
                load_warp_consts(wc, consts + seg, lane);
                cur = seg;
            }

            double acc[NA];
#pragma unroll
            for (int a = 0; a < NA; ++a) acc[a] = 0.0;
            double prod = 1.0;   // unweighted: product of mantissas of P ...
            int esum = 0;        // ... and sum of exponents (log_mul)

            // Events are taken kSub rows at a time (lane l: l + 32 i).  Those with t <= tcut
            // (about a fifth of them) need the Gaussian and erfcx: slow_rows.
            const int64_t tbase = ev0 + (tile - t0) * kTile;
            if constexpr (GRAD)
                solo_tile<Model<KIND, CACHED>, WEIGHTED>(wc, &mt, cols, tbase, ev1, sbuf, wbuf, lane, acc, &prod, &esum);
            else
                plain_rows<KIND, GRAD, CACHED, WEIGHTED>(wc, &mt, cols, 0, tile_rows(tbase, ev1), tbase, ev1, sbuf, lane,
                                                         acc, &prod, &esum);
            acc[0] += log_of(prod, esum, &mt);
            const double share = warp_butterfly<NA>(acc, lane);
            // the group and segment levels; the warp that completes the
            // segment writes its NLL and gradient
            if (!tile_commit<NA>(share, lane, tile, t0, t1, seg, partials, gcount, counters, acc)) continue;
            finalize<KIND, GRAD, CACHED>(wc, acc, n_par, out + (size_t)seg * out_stride, lane);
            if (lane == 0) counters[seg] = 0u;
        }
    }
    work_done(work, lane);
}

// seg_tiles[s] = sum_{r<s} tiles(r), tiles(r) = ceil(size_r / kTile) for an active
// segment (0 when active[r] == 0), one block: sequential per thread over a
// contiguous run of segments, then a block scan of the run totals.
__global__ void seg_tiles_kernel(const int64_t* __restrict__ seg_begin, const int64_t* __restrict__ seg_end,
                                 const int* __restrict__ active, int n_seg, int64_t n,
                                 int64_t* __restrict__ seg_tiles) {
    __shared__ int64_t run[1024];
    const int nt = blockDim.x;
    const int per = (n_seg + nt - 1) / nt;
    const int b = threadIdx.x * per;
    const int e = min(n_seg, b + per);
    auto tiles = [&](int s) -> int64_t {
        if (active && !active[s]) return 0;
        const int64_t lo = clamp_off(seg_begin[s], n);
        int64_t hi = clamp_off(seg_end[s], n);
        if (hi < lo) hi = lo;
        return (hi - lo + kTile - 1) / kTile;
    };
    int64_t sum = 0;
    for (int s = b; s < e; ++s) sum += tiles(s);
    run[threadIdx.x] = sum;
    __syncthreads();
    for (int d = 1; d < nt; d <<= 1) {
        const int64_t v = threadIdx.x >= d ? run[threadIdx.x - d] : 0;
        __syncthreads();
        run[threadIdx.x] += v;
        __syncthreads();
    }
    int64_t acc = threadIdx.x ? run[threadIdx.x - 1] : 0;
    for (int s = b; s < e; ++s) {
        seg_tiles[s] = acc;
        acc += tiles(s);
    }
    if (threadIdx.x == nt - 1) seg_tiles[n_seg] = run[nt - 1];
}

template <int KIND, bool GRAD, bool CACHED, bool WEIGHTED>
ipa_status launch_t(const Cols& cols, int64_t n, const int64_t* seg_begin, const int64_t* seg_end,
                    const int64_t* seg_tiles, int n_seg, const Consts* consts, Scratch* sc, double* out,
                    int n_par, cudaStream_t st, const LaunchCfg* force) {
    const bool single = seg_begin == nullptr;
    const int64_t tiles = tile_estimate(n, n_seg);
    const LaunchCfg cfg = force ? *force : launch_cfg(KIND, GRAD, CACHED, n_seg > 1, tiles);
    if constexpr (GRAD) {
        if (launch_team_ok<Model<KIND, CACHED>, WEIGHTED>(cfg, n, n_seg))
            return launch_team<Model<KIND, CACHED>, WEIGHTED>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out,
                                                      n_par, tiles, st);
    }
    const int W = cfg.warps_per_block >= 1 && cfg.warps_per_block <= kMaxWarps ? cfg.warps_per_block : 1;
    const int K = cfg.tiles_per_take >= 1 ? cfg.tiles_per_take : 1;
    const size_t smem = (size_t)W * (sizeof(Consts) + kSub * 32 * (sizeof(double2) + (GRAD && WEIGHTED ? sizeof(double) : 0)));
    // resident blocks per SM for each block size (cached per device and variant)
    static int occ[64][kMaxWarps + 1] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    int& per_sm = occ[dev & 63][W];
    if (per_sm == 0) {
        int v = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &v, nll_kernel<KIND, GRAD, CACHED, WEIGHTED>, 32 * W, smem);
        per_sm = e == cudaSuccess && v >= 1 ? v : 1;
    }
    const int64_t grid = launch_grid(cfg, W, K, per_sm, tiles, single);
    // programmatic dependent launch: blocks may start (and load their tables)
    // while the constants kernel that precedes every launch is still running
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)grid);
    lc.blockDim = dim3(32u * W);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = 1;
    return cuda_fail(cudaLaunchKernelEx(&lc, nll_kernel<KIND, GRAD, CACHED, WEIGHTED>, cols, n, seg_begin, seg_end,
                                        seg_tiles, n_seg, consts, sc->partials, sc->counters, sc->gcount, sc->work,
                                        out, n_par, K),
                     "likelihood kernel launch");
}

}  // namespace

ipa_status launch_seg_tiles(const int64_t* seg_begin, const int64_t* seg_end, const int* active, int n_seg,
                            int64_t n, int64_t* seg_tiles, cudaStream_t st) {
    seg_tiles_kernel<<<1, 1024, 0, st>>>(seg_begin, seg_end, active, n_seg, n, seg_tiles);
    return cuda_fail(cudaGetLastError(), "segment tiling kernel launch");
}

// Kernel variant for a launch: model, gradient, cached basis, weights.
template <int KIND, bool GRAD, bool CACHED>
ipa_status launch_w(const Cols& cols, int64_t n, const int64_t* seg_begin, const int64_t* seg_end,
                    const int64_t* seg_tiles, int n_seg, const Consts* consts, Scratch* sc, double* out,
                    int n_par, cudaStream_t st, const LaunchCfg* cfg) {
    if (cols.w)
        return launch_t<KIND, GRAD, CACHED, true>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out,
                                                  n_par, st, cfg);
    return launch_t<KIND, GRAD, CACHED, false>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out,
                                               n_par, st, cfg);
}

ipa_status launch_nll(const ModelDev& m, bool grad, const Cols& cols, int64_t n,
                      const int64_t* seg_begin, const int64_t* seg_end, const int64_t* seg_tiles, int n_seg,
                      const Consts* consts, Scratch* sc, double* out, cudaStream_t st, const LaunchCfg* cfg) {
    const int P = m.n_par;
    if (m.kind == IPA_MODEL_TAGGED1D)
        return launch_tag_nll(m, grad, cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, st, cfg);
    if (m.kind == IPA_MODEL_PHIS)
        return launch_phis_nll(m, grad, cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, st, cfg);
    if (m.kind == IPA_MODEL_TIME1D)
        return grad ? launch_w<IPA_MODEL_TIME1D, true, false>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, P, st, cfg)
                    : launch_w<IPA_MODEL_TIME1D, false, false>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, P, st, cfg);
    if (cols.fk)
        return grad ? launch_w<IPA_MODEL_ANGTIME4D, true, true>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, P, st, cfg)
                    : launch_w<IPA_MODEL_ANGTIME4D, false, true>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, P, st, cfg);
    return grad ? launch_w<IPA_MODEL_ANGTIME4D, true, false>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, P, st, cfg)
                : launch_w<IPA_MODEL_ANGTIME4D, false, false>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, P, st, cfg);
}

// f_k = c_k f'_k for every event (the cached angular basis).
__global__ void __launch_bounds__(kNllBlock)
basis_kernel(const double* __restrict__ ck, const double* __restrict__ cl, const double* __restrict__ phi,
             int64_t n, double* __restrict__ fk, int64_t stride) {
    __shared__ MathTables mt;
    load_math_tables(&mt);
    __syncthreads();
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        double f[10];
        basis_unscaled(__ldg(ck + e), __ldg(cl + e), __ldg(phi + e), &mt, f);
#pragma unroll
        for (int k = 0; k < 10; ++k) fk[k * stride + e] = kBasisScale[k] * f[k];
    }
}

}  // namespace ipa

extern "C" ipa_status ipa_angular_basis(const ipa_model* model, const ipa_events* ev, double* fk_dev,
                                        int64_t stride, void* stream) {
    using namespace ipa;
    ipa_status st = check_model(model);
    if (st != IPA_OK) return st;
    if (model->kind != IPA_MODEL_ANGTIME4D && model->kind != IPA_MODEL_PHIS) {
        set_error("ipa_angular_basis: the model has no angles");
        return IPA_ERR_ARG;
    }
    ipa_events plain = *ev;
    plain.fk = nullptr;
    if ((st = check_events(model, &plain)) != IPA_OK) return st;
    if (!fk_dev || (reinterpret_cast<uintptr_t>(fk_dev) & 15u) || stride < ev->n || (stride & 1)) {
        set_error("ipa_angular_basis: 16-byte aligned output with an even stride >= n required");
        return IPA_ERR_ARG;
    }
    if (ev->n == 0) return IPA_OK;
    const int64_t blocks = (ev->n + kNllBlock - 1) / kNllBlock;
    const int grid = (int)(blocks < 4 * sm_count() * 4 ? blocks : 4 * sm_count() * 4);
    basis_kernel<<<grid, kNllBlock, 0, static_cast<cudaStream_t>(stream)>>>(ev->ck, ev->cl, ev->phi, ev->n, fk_dev,
                                                                            stride);
    return cuda_fail(cudaGetLastError(), "angular basis kernel launch");
}

namespace ipa {

namespace {

ipa_status run(const ipa_model* model, const ipa_events* ev, const int64_t* seg_off, int n_seg,
               const double* theta, double* out, bool grad, void* stream) {
    ipa_status st = check_model(model);
    if (st != IPA_OK) return st;
    if ((st = check_events(model, ev)) != IPA_OK) return st;
    if (!theta || !out) {
        set_error("theta and out must be device pointers");
        return IPA_ERR_ARG;
    }
    if (n_seg < 1) {
        set_error("n_seg must be >= 1");
        return IPA_ERR_ARG;
    }
    if (seg_off == nullptr && n_seg != 1) {
        set_error("segment offsets are required for n_seg > 1");
        return IPA_ERR_ARG;
    }
    const int64_t tiles = (ev->n + kTile - 1) / kTile + n_seg;
    Scratch* sc = nullptr;
    if ((st = scratch_get(tiles, n_seg + 1, &sc)) != IPA_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const ModelDev m{model->kind, model->n_par, model->t_lo, model->t_hi};
    if ((st = launch_consts(m, theta, n_seg, sc->consts, s)) != IPA_OK) return st;
    if (seg_off) {
        if ((st = launch_seg_tiles(seg_off, seg_off + 1, nullptr, n_seg, ev->n, sc->seg_tiles, s)) != IPA_OK)
            return st;
    }
    const Cols cols{ev->t, ev->ck, ev->cl, ev->phi, ev->w, ev->fk, ev->fk_stride, ev->q};
    return launch_nll(m, grad, cols, ev->n, seg_off, seg_off ? seg_off + 1 : nullptr,
                      seg_off ? sc->seg_tiles : nullptr, n_seg, sc->consts, sc, out, s);
}

// ---- event-sharded likelihood ----
// After a single-segment launch, group g's reduced partial (the sums of its 32
// tiles) sits in the slot of its first tile, g * kGroupTiles.  Copy them out,
// n_groups x na doubles, in group order.
__global__ void group_partials_kernel(const double* __restrict__ partials, int na, int64_t n_groups,
                                      double* __restrict__ out) {
    const int64_t total = n_groups * na;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = i / na;
        out[i] = __ldcg(partials + (g * kGroupTiles) * na + (i - g * na));
    }
}

// The last level of the kernel's reduction (lane l adds groups l, l + 32, ...
// in order, then the butterfly) and the gradient contraction, over group
// partials gathered from several launches: one warp.
template <int KIND, bool CACHED>
__global__ void combine_kernel(const double* __restrict__ groups, int64_t n_groups, const Consts* __restrict__ consts,
                               int n_par, double* __restrict__ out) {
    constexpr int NA = n_acc(KIND, true);
    const int lane = threadIdx.x & 31;
    if (n_groups == 0) {
        for (int j = lane; j < 1 + n_par; j += 32) out[j] = 0.0;
        return;
    }
    double acc[NA];
    gather_butterfly<NA>(reduce_partials<NA>(groups, 0, n_groups, 1, lane), acc);
    finalize<KIND, true, CACHED>(consts[0], acc, n_par, out, lane);
}

}  // namespace
}  // namespace ipa

extern "C" ipa_status ipa_nll(const ipa_model* model, const ipa_events* ev, const double* theta_dev,
                              double* out_dev, void* stream) {
    return ipa::run(model, ev, nullptr, 1, theta_dev, out_dev, false, stream);
}

extern "C" ipa_status ipa_nll_grad(const ipa_model* model, const ipa_events* ev,
                                   const double* theta_dev, double* out_dev, void* stream) {
    return ipa::run(model, ev, nullptr, 1, theta_dev, out_dev, true, stream);
}

extern "C" ipa_status ipa_nll_grad_segmented(const ipa_model* model, const ipa_events* ev,
                                             const int64_t* seg_off_dev, int32_t n_seg,
                                             const double* theta_dev, double* out_dev,
                                             void* stream) {
    if (!seg_off_dev) {
        ipa::set_error("seg_off_dev must not be NULL");
        return IPA_ERR_ARG;
    }
    return ipa::run(model, ev, seg_off_dev, n_seg, theta_dev, out_dev, true, stream);
}


// Group partials of a single-segment call over n events: ceil(n / 16384).
static int64_t shard_groups(int64_t n) {
    const int64_t tiles = (n + ipa::kTile - 1) / ipa::kTile;
    return (tiles + ipa::kGroupTiles - 1) / ipa::kGroupTiles;
}

extern "C" ipa_status ipa_shard_width(const ipa_model* model, int32_t* width) {
    ipa_status st = ipa::check_model(model);
    if (st != IPA_OK) return st;
    if (!width) {
        ipa::set_error("ipa_shard_width: width is NULL");
        return IPA_ERR_ARG;
    }
    *width = ipa::n_acc(model->kind, true);
    return IPA_OK;
}

extern "C" ipa_status ipa_nll_grad_shard(const ipa_model* model, const ipa_events* ev, const double* theta_dev,
                                         double* out_dev, double* groups_dev, void* stream) {
    using namespace ipa;
    if (!groups_dev && ev && ev->n > 0) {
        set_error("ipa_nll_grad_shard: groups_dev is NULL");
        return IPA_ERR_ARG;
    }
    ipa_status st = run(model, ev, nullptr, 1, theta_dev, out_dev, true, stream);
    if (st != IPA_OK || ev->n == 0) return st;
    Scratch* sc = nullptr;
    if ((st = scratch_get((ev->n + kTile - 1) / kTile + 1, 2, &sc)) != IPA_OK) return st;
    const int na = n_acc(model->kind, true);
    const int64_t ng = shard_groups(ev->n);
    const int64_t blocks = (ng * na + 255) / 256;
    group_partials_kernel<<<(unsigned)(blocks < 1024 ? blocks : 1024), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        sc->partials, na, ng, groups_dev);
    return cuda_fail(cudaGetLastError(), "group partials copy");
}

extern "C" ipa_status ipa_nll_grad_combine(const ipa_model* model, const double* theta_dev, const double* groups_dev,
                                           int64_t n_groups, int32_t cached, double* out_dev, void* stream) {
    using namespace ipa;
    ipa_status st = check_model(model);
    if (st != IPA_OK) return st;
    if (!theta_dev || !out_dev || n_groups < 0 || (n_groups > 0 && !groups_dev)) {
        set_error("ipa_nll_grad_combine: bad arguments");
        return IPA_ERR_ARG;
    }
    if (cached && model->kind != IPA_MODEL_ANGTIME4D && model->kind != IPA_MODEL_PHIS) {
        set_error("ipa_nll_grad_combine: only models with angles have a cached basis");
        return IPA_ERR_ARG;
    }
    Scratch* sc = nullptr;
    if ((st = scratch_get(1, 2, &sc)) != IPA_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const ModelDev m{model->kind, model->n_par, model->t_lo, model->t_hi};
    if ((st = launch_consts(m, theta_dev, 1, sc->consts, s)) != IPA_OK) return st;
    const int P = model->n_par;
    switch (model->kind) {
    case IPA_MODEL_TIME1D:
        combine_kernel<IPA_MODEL_TIME1D, false><<<1, 32, 0, s>>>(groups_dev, n_groups, sc->consts, P, out_dev);
        break;
    case IPA_MODEL_ANGTIME4D:
        if (cached)
            combine_kernel<IPA_MODEL_ANGTIME4D, true><<<1, 32, 0, s>>>(groups_dev, n_groups, sc->consts, P, out_dev);
        else
            combine_kernel<IPA_MODEL_ANGTIME4D, false><<<1, 32, 0, s>>>(groups_dev, n_groups, sc->consts, P, out_dev);
        break;
    case IPA_MODEL_TAGGED1D:
        return launch_tag_combine(groups_dev, n_groups, sc->consts, P, out_dev, s);
    default:
        return launch_phis_combine(groups_dev, n_groups, cached != 0, sc->consts, P, out_dev, s);
    }
    return cuda_fail(cudaGetLastError(), "combine kernel launch");
}
