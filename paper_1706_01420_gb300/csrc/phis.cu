// Hot path of the full time-dependent angular model with tagging (the phi_s
// fit of Sec. 4; formulas in ipanema.h): constants, the likelihood with its
// fused gradient, and the deterministic reduction.
//
// Coefficient form.  Each angular term k is a bilinear b_k = conj(A_i) A_j of
// transversity amplitudes with CP eigenvalues eta_i, eta_j; with the time
// evolution its tag-mixed rate is a combination of four convolved time
// functions, G = (g_L, g_H, q Re g_c, q Im g_c) (g_c = g(tau; Gamma - i Dm)):
//   rate(t, Omega, q) = sum_k f_k sum_j C_kj G_j,
// where, with c, s = cos, sin phi_s and D = 1 - 2 omega, for
//   eta_i = eta_j = eta:   part(b) (1 + eta c)/2, part(b) (1 - eta c)/2, 0, D eta s part(b),
//   eta_i = -eta_j, eta = eta_j, real part:
//       eta s Im b / 2, -eta s Im b / 2, D Re b, -D eta c Im b,
//   imaginary part:
//       -eta s Re b / 2, eta s Re b / 2, D Im b, D eta c Re b
// (part = Re or Im as the term takes; the products of g+- are written out
// in ipanema.h).
//
// The kernel does not evaluate the 40 entries of C: the terms share four time
// functions.  A term whose amplitudes have the same CP eigenvalue takes
// T+ or T-, a mixed one U and V,
//   T+- = (gL + gH)/2 +- [c (gL - gH)/2 + D s q Im g_c],
//   U = s (gL - gH)/2 - D c q Im g_c,   V = D q Re g_c:
//   equal: part(b) T_eta;  real mixed: eta Im b U + Re b V;  imaginary mixed: -eta Re b U + Im b V.
// Per event: the ten f'_k (integer pipe), the four convolutions (as in
// tagged.cu), four angular sums F+, F-, FU, FV (14 products instead of 40), and
// P = F+ T+ + F- T- + FU U + FV V + cb regrouped by convolution.
//
// Gradient.  The amplitude and C_SP parameters need the 14 sums of r f'_k times
// its time functions (40 before).  phi_s: dT+- = -+U, dU = (T+ - T-)/2, one
// sum of (F- - F+) U + FU dU.  The mistag needs the tag-odd part of the rate, a
// sum the time parameters need anyway.  These are linear in 14 sums (r times
// the rate's part of each convolution, plain and times tau, and the Gaussian's):
// dg/dz = (z sigma^2 - tau) g - sigma^2 G, dg/dsigma = z^2 sigma g - (z sigma +
// tau/sigma) G, dg/dtau = -z g + G.  With the log and Q = sum r: 31 sums, one per
// lane once reduced (47 before).
//
// Bound: the FP64 pipe.  Fewer operations per event and registers for three
// blocks per SM in place of two are the gain over the 40-product form; figures at
// phis_kernel.
#include <math.h>
#include <stddef.h>

#include "accept_reject.cuh"
#include "angular.cuh"
#include "consts.cuh"
#include "conv32.cuh"
#include "faddeeva.cuh"
#include "fp64_math.cuh"
#include "int_math.cuh"
#include "ipa_internal.cuh"
#include "philox.cuh"
#include "phis_consts.cuh"
#include "tagged.cuh"
#include "team_tile.cuh"
#include "tile_reduce.cuh"

namespace ipa {
namespace {

constexpr int kMaxWarps = 8;
constexpr int kRow = n_acc(IPA_MODEL_PHIS, true);   // doubles per tile or group partial (the width of a shard's rows)
constexpr int kNA = 31;          // accumulators with the gradient; the row's other entries are zero
static_assert(kNA <= 32 && kNA <= kRow && kRow <= kMaxAcc, "one accumulator per lane, rows in the scratch");
// Accumulators: the log, Q = sum r, the equal terms' sums (order kEq), the mixed
// terms' sums with U and with V / D (order kMix), phi_s, then the time sums.
enum {
    kLog, kQ, kE, kMU = kE + 6, kMV = kMU + 4, kPhi = kMV + 4,
    kL0, kL1, kH0, kH1,          // r FwL gL, times tau; H likewise
    kY10, kY11, kY20, kY21,      // r Y1, r Y2 (the tag-odd part and its quadrature), times tau
    kGa, kGb, kGc, kGd,          // r Gx times FwL, FwH, q FV, q X
    kGt1, kGt2,                  // r tau Gx times FwL + FwH, q FV
    kEnd
};
static_assert(kEnd == kNA, "accumulator list");
__device__ const int kEq[6] = {0, 1, 4, 2, 6, 8};    // eta = +1 (three), eta = -1 (three)
__device__ const int kMix[4] = {3, 5, 7, 9};
__device__ const double kEta[4] = {1.0, 1.0, -1.0, -1.0};

// (i, j, imaginary part?) of the ten bilinears conj(A_i) A_j (0, para, perp, S)
__device__ const int kPairI[10] = {0, 1, 2, 1, 0, 0, 3, 3, 3, 3};
__device__ const int kPairJ[10] = {0, 1, 2, 2, 1, 2, 3, 1, 2, 0};
__device__ const int kPairIm[10] = {0, 0, 0, 1, 0, 1, 0, 0, 1, 0};

// Row factor: C_SP for the S-P interference terms, 1 otherwise.
__device__ __forceinline__ double row_scale(const PhisConsts& c, int k) { return k >= 7 ? c.csp : 1.0; }

// Row k of C from part(b) pieces: pr = Re b, pi = Im b.  Every entry is a
// product of part(b), one of (one, c, s) and of wu (untagged entries) or wt
// (tagged entries, D), so that with (one, c, s) = (1, cos, sin phi_s) and
// (wu, wt) = (1, D) it is C itself, with (0, -sin, cos) its derivative in
// phi_s, and with (wu, wt) = (0, -2) its derivative in omega.
__device__ inline void c_row(int k, double pr, double pi, double one, double c, double s, double wu, double wt,
                             double* out) {
    const double ei = kEta[kPairI[k]], ej = kEta[kPairJ[k]];
    if (ei == ej) {
        const double p = kPairIm[k] ? pi : pr;
        out[0] = wu * 0.5 * p * (one + ej * c);
        out[1] = wu * 0.5 * p * (one - ej * c);
        out[2] = 0.0;
        out[3] = wt * ej * s * p;
    } else if (!kPairIm[k]) {
        out[0] = wu * 0.5 * ej * s * pi;
        out[1] = -wu * 0.5 * ej * s * pi;
        out[2] = wt * one * pr;
        out[3] = -wt * ej * c * pi;
    } else {
        out[0] = -wu * 0.5 * ej * s * pr;
        out[1] = wu * 0.5 * ej * s * pr;
        out[2] = wt * one * pi;
        out[3] = wt * ej * c * pr;
    }
}

// The ten f'_k on the integer pipe, rounded once to double (1e6 events: 313 us with
// 14-instruction 64-bit products, 300 us with those of fast_fixed.cuh), in FP64 near
// |cos| = 1.
__device__ __forceinline__ void phis_basis(double ck, double cl, double phi, const MathTables* mt, double f[10]) {
    if (fx_angles_ok(ck, cl, phi)) {
        long long g[10];
        fx_basis(ck, cl, phi, mt, g);
        const long long F[10] = {g[0] - g[2], g[1] - g[3], g[1] - g[2] + g[3], g[4], g[5],
                                 g[6], g[0], g[7], g[8], g[9]};
#pragma unroll
        for (int k = 0; k < 10; ++k) f[k] = fx_to_double(F[k], 0);
    } else {
        basis_unscaled(ck, cl, phi, mt, f);
    }
}

// Per-warp copy: the record and the coefficients of the angular sums, with cs / 4
// (P from the doubled convolutions, and the halves of T and U), the basis factor
// c_k (1 for a cached basis) and C_SP folded in.
struct PhisWarp {
    PhisConsts c;
    double eq[6], mu[4], mv[4];
    double D2, D2s, D2c;      // 2 D, 2 D s, 2 D c
    // the same in fixed point (phis_event_fast): eq, mu, mv with max in [1/8, 1/4) at 2^-hexp; c and s
    // (Q62); rtop: scale of the angular sums' factors at unit weight (2^11 typical ones, 2^(rtop - 2))
    int2 fe[6], fu[4], fv[4], fc, fs;
    int hexp, rtop, fixed, pad_;
};

static_assert(offsetof(PhisWarp, fs) == offsetof(PhisWarp, fe) + 15 * sizeof(int2), "one run of coefficients");

__device__ __forceinline__ void phis_coefficients(PhisWarp& pw, bool cached, int lane) {
    const PhisConsts& c = pw.c;
    int ex = 0;               // largest exponent field of the coefficients
    if (lane < 10) {
        const int k = lane < 6 ? kEq[lane] : kMix[lane - 6];
        const double sc = 0.25 * c.cs * row_scale(c, k) * (cached ? 1.0 : kBasisScale[k]);
        const double re = kPairIm[k] ? c.bi[k] : c.br[k];
        if (lane < 6) {
            pw.eq[lane] = sc * re;
            ex = exponent_field(pw.eq[lane]);
        } else {
            const double ej = kEta[kPairJ[k]];
            pw.mu[lane - 6] = sc * (kPairIm[k] ? -ej * c.br[k] : ej * c.bi[k]);
            pw.mv[lane - 6] = sc * re;
            ex = max(exponent_field(pw.mu[lane - 6]), exponent_field(pw.mv[lane - 6]));
        }
    } else if (lane == 10) {
        pw.D2 = 2.0 * c.D;
        pw.D2s = 2.0 * c.D * c.s;
        pw.D2c = 2.0 * c.D * c.c;
    }
    ex = __reduce_max_sync(0xffffffffu, ex);
    const int up = 1020 - ex;                             // max|coefficient| 2^up in [1/8, 1/4)
    const bool ok = up >= -64 && up <= 900 && abs_below(c.c, 1.5) && abs_below(c.s, 1.5);
    const double sc = __longlong_as_double((long long)((ok ? up : 0) + 1023) << 52);
    if (lane < 16 && ok) {
        const double x = lane < 6 ? pw.eq[lane] : (lane < 10 ? pw.mu[lane - 6] : (lane < 14 ? pw.mv[lane - 10] : (lane == 14 ? c.c : c.s)));
        const Fx v = fx(fx_signed(lane < 14 ? x * sc : x, 1));
        pw.fe[lane] = make_int2(v.h, v.l);                // fe, fu, fv, fc, fs are contiguous
    } else if (lane == 16) {
        // a typical r T is near 1 / max(max|coefficient|, cb / 4)
        const int ea = ok ? -up - 3 : -1023, eb = exponent_field(c.cb) - 1025;
        const int e = ea > eb ? ea : eb;
        pw.rtop = 13 + (e < -900 ? 900 : -e);
        pw.hexp = 2 - (ok ? up : 0);
        pw.fixed = ok;
    }
}

// One event: log term and, with GRAD, the sums.  The convolutions are doubled
// (as in tagged.cu).
template <bool GRAD, bool WEIGHTED>
__device__ __forceinline__ void phis_event(const PhisWarp& pw, const MathTables* mt, double t, double q, double w,
                                           const double* f, const TagSlow& sl, double* acc, double* prod,
                                           int* esum) {
    const PhisConsts& c = pw.c;
    const double tau = t - c.mu;
    const TimeValues v = time_values(c, t, tau, mt);
    const long long bH = __double_as_longlong(sl.xH), bL = __double_as_longlong(sl.xL);
    const long long bG = __double_as_longlong(sl.gx);
    const double H = bH < 0 ? -sl.xH : v.H - sl.xH;
    const double L = bL < 0 ? -sl.xL : v.L - sl.xL;
    const double Cr = q * (bG < 0 ? sl.wr : fma(v.C, v.cn, -sl.wr));
    const double Ci = q * (bG < 0 ? sl.wi : fma(v.C, v.sn, -sl.wi));
    // F+, F-, FU, FV; the rate's coefficients of L and H, and of D2 Ci (X)
    const double Fp = fma(pw.eq[2], f[4], fma(pw.eq[1], f[1], pw.eq[0] * f[0]));
    const double Fm = fma(pw.eq[5], f[8], fma(pw.eq[4], f[6], pw.eq[3] * f[2]));
    const double FU = fma(pw.mu[3], f[9], fma(pw.mu[2], f[7], fma(pw.mu[1], f[5], pw.mu[0] * f[3])));
    const double FV = fma(pw.mv[3], f[9], fma(pw.mv[2], f[7], fma(pw.mv[1], f[5], pw.mv[0] * f[3])));
    const double Fs = Fp + Fm, Fd = Fp - Fm;
    const double hd = fma(c.c, Fd, c.s * FU);
    const double FL = Fs + hd, FH = Fs - hd;
    const double X = fma(c.s, Fd, -(c.c * FU));
    const double Y1 = fma(Cr, FV, Ci * X);
    const double P = fma(FL, L, fma(FH, H, fma(pw.D2, Y1, c.cb)));
    if (WEIGHTED && __double_as_longlong(w) != 0x3FF0000000000000ll)
        acc[kLog] = fma(w, log_fast(P, mt), acc[kLog]);
    else
        log_mul(P, prod, esum);
    if (!GRAD) return;
    const double r = WEIGHTED ? w * rcp_newton(P) : rcp_newton(P);
    acc[kQ] += r;
    const double sG = L + H, dG = L - H;
    const double m = fma(c.c, dG, pw.D2s * Ci);       // (T+ - T-)/2 and dU/dphi_s, four times
    const double rp = r * (sG + m), rm = r * (sG - m);
    const double u = fma(c.s, dG, -(pw.D2c * Ci));    // U, four times
    const double ru = r * u, rv = r * Cr;
    acc[kE + 0] = fma(rp, f[0], acc[kE + 0]);
    acc[kE + 1] = fma(rp, f[1], acc[kE + 1]);
    acc[kE + 2] = fma(rp, f[4], acc[kE + 2]);
    acc[kE + 3] = fma(rm, f[2], acc[kE + 3]);
    acc[kE + 4] = fma(rm, f[6], acc[kE + 4]);
    acc[kE + 5] = fma(rm, f[8], acc[kE + 5]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        acc[kMU + i] = fma(ru, f[3 + 2 * i], acc[kMU + i]);
        acc[kMV + i] = fma(rv, f[3 + 2 * i], acc[kMV + i]);
    }
    acc[kPhi] = fma(r * m, FU, fma(-ru, Fd, acc[kPhi]));
    const double hL = (r * FL) * L, hH = (r * FH) * H;
    acc[kL0] += hL;
    acc[kL1] = fma(hL, tau, acc[kL1]);
    acc[kH0] += hH;
    acc[kH1] = fma(hH, tau, acc[kH1]);
    const double y1 = r * Y1, y2 = r * fma(Ci, FV, -(Cr * X));
    acc[kY10] += y1;
    acc[kY11] = fma(y1, tau, acc[kY11]);
    acc[kY20] += y2;
    acc[kY21] = fma(y2, tau, acc[kY21]);
    const double g = r * __longlong_as_double(bG & 0x7FFFFFFFFFFFFFFFll), gq = g * q, gt = g * tau;
    acc[kGa] = fma(g, FL, acc[kGa]);
    acc[kGb] = fma(g, FH, acc[kGb]);
    acc[kGc] = fma(gq, FV, acc[kGc]);
    acc[kGd] = fma(gq, X, acc[kGd]);
    acc[kGt1] = fma(gt, Fs, acc[kGt1]);               // (FL + FH) / 2
    acc[kGt2] = fma(gq * tau, FV, acc[kGt2]);
}

// ---- the fixed-point form of an event's angular part (NLL + gradient) ----
// As in the 4D kernel's fast rows (nll.cu): the ten f'_k (Q62), F+, F-, FU, FV and what is linear
// in them on the integer pipe, and the 14 angular sums as 64-bit integers: the factors r T+, r T-,
// r U and r C are converted once per event at a scale that follows the segment's typical r T and
// the largest weight of the warp's rows (unit 2^-48 of a typical term, 0.41 units rms per
// event).  The rest is FP64.  The warp's rows are redone by phis_event where some P lies outside
// the Newton reciprocal's range, some factor above its scale or all of them far below it.
// FP64 instructions per event: 92 -> 57; 1e6 events 299 -> 248 us (FP64 unit busy 77 -> 68 %).

// The f'_k in Q62 near |cos| = 1 (rare).  False where one of them does not fit (angles that
// are NaN or infinite, |cos| > 1): the rows are left to phis_event.
__device__ __noinline__ bool phis_basis_wide(double ck, double cl, double phi, const MathTables* mt, long long F[10]) {
    double f[10];
    basis_unscaled(ck, cl, phi, mt, f);
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 10; ++k) {
        ok = ok && fits_q62(f[k]);
        F[k] = to_q62_nb(f[k]);
    }
    return ok;
}

// One event: FP64 sums into acc (as phis_event), the angular sums (kE .. kMV + 3) into S.
template <bool WEIGHTED, bool CACHED>
__device__ __forceinline__ void phis_event_fast(const PhisWarp& pw, const MathTables* mt, const Cols& cols, int64_t e,
                                                const TagSlow& sl, int top, double* acc, long long* S, double* prod,
                                                int* esum, bool* bad) {
    const PhisConsts& c = pw.c;
    const double t = __ldg(cols.t + e), q = __ldg(cols.q + e);
    const double w = WEIGHTED ? __ldg(cols.w + e) : 1.0;
    long long F[10];
    if (CACHED) {
#pragma unroll
        for (int k = 0; k < 10; ++k) {
            const double f = __ldg(cols.fk + k * cols.fk_stride + e);
            *bad |= !fits_q62(f);
            F[k] = fx_signed(f, 1);
        }
    } else {
        const double ck = __ldg(cols.ck + e), cl = __ldg(cols.cl + e), phi = __ldg(cols.phi + e);
        long long g[10];
        fx_basis(ck, cl, phi, mt, g);
        F[0] = g[0] - g[2];
        F[1] = g[1] - g[3];
        F[2] = F[1] - g[2] + g[3] + g[3];
        F[3] = g[4];
        F[4] = g[5];
        F[5] = g[6];
        F[6] = g[0];
        F[7] = g[7];
        F[8] = g[8];
        F[9] = g[9];
        if (!fx_angles_ok(ck, cl, phi)) {
            long long x[10];                             // (a copy, so that F itself stays in registers)
            *bad |= !phis_basis_wide(ck, cl, phi, mt, x);
#pragma unroll
            for (int k = 0; k < 10; ++k) F[k] = x[k];
        }
    }
    const auto K = [](const int2& a) { return Fx{a.x, a.y}; };
    const long long fp = fx_mad(K(pw.fe[2]), fx(F[4]), fx_mad(K(pw.fe[1]), fx(F[1]), fx_mad(K(pw.fe[0]), fx(F[0]), 0)));
    const long long fm = fx_mad(K(pw.fe[5]), fx(F[8]), fx_mad(K(pw.fe[4]), fx(F[6]), fx_mad(K(pw.fe[3]), fx(F[2]), 0)));
    long long fu = 0, fv = 0;                             // Q60, as fp and fm
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        fu = fx_mad(K(pw.fu[i]), fx(F[3 + 2 * i]), fu);
        fv = fx_mad(K(pw.fv[i]), fx(F[3 + 2 * i]), fv);
    }
    const long long fsum = fp + fm, fdif = fp - fm;
    const Fx D = fx(fdif), U = fx(fu);
    const long long hd = fx_mad(K(pw.fc), D, fx_mad(K(pw.fs), U, 0)) << 2;
    const long long xx = (fx_mad(K(pw.fs), D, 0) - fx_mad(K(pw.fc), U, 0)) << 2;
    const double FL = fx_to_double(fsum + hd, pw.hexp), FH = fx_to_double(fsum - hd, pw.hexp);
    const double X = fx_to_double(xx, pw.hexp), FV = fx_to_double(fv, pw.hexp);
    const double FU = fx_to_double(fu, pw.hexp), Fd = fx_to_double(fdif, pw.hexp);

    const double tau = t - c.mu;
    const TimeValues v = time_values(c, t, tau, mt);
    const long long bH = __double_as_longlong(sl.xH), bL = __double_as_longlong(sl.xL);
    const long long bG = __double_as_longlong(sl.gx);
    const double H = bH < 0 ? -sl.xH : v.H - sl.xH;
    const double L = bL < 0 ? -sl.xL : v.L - sl.xL;
    const double Cr = q * (bG < 0 ? sl.wr : fma(v.C, v.cn, -sl.wr));
    const double Ci = q * (bG < 0 ? sl.wi : fma(v.C, v.sn, -sl.wi));
    const double Y1 = fma(Cr, FV, Ci * X);
    const double P = fma(FL, L, fma(FH, H, fma(pw.D2, Y1, c.cb)));
    *bad |= (unsigned long long)(__double_as_longlong(P) - 0x3820000000000000ll) >= 0x0FB0000000000000ull;
    if (WEIGHTED) {
        const bool one = __double_as_longlong(w) == 0x3FF0000000000000ll;
        acc[kLog] = fma(one ? 0.0 : w, fx_to_double(fx_log(P, mt), 6), acc[kLog]);
        log_mul_nb(one ? P : 1.0, prod, esum);
    } else {
        log_mul_nb(P, prod, esum);
    }
    const double r = WEIGHTED ? w * rcp_newton_nb(P) : rcp_newton_nb(P);
    acc[kQ] += r;
    const double sG = L + H, dG = L - H;
    const double m = fma(c.c, dG, pw.D2s * Ci);
    const double u = fma(c.s, dG, -(pw.D2c * Ci));
    const double ru = r * u;
    {
        const double x[4] = {r * (sG + m), r * (sG - m), ru, r * Cr};
        Fx A[4];
        int one[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            *bad |= exponent_field(x[i]) > 1023 - 3 + top;
            const long long a = fx_odd(x[i], top);
            one[i] = a != 0;
            A[i] = fx(a);
        }
        S[0] = fx_mad1(A[0], fx(F[0]), S[0], one[0]);
        S[1] = fx_mad1(A[0], fx(F[1]), S[1], one[0]);
        S[2] = fx_mad1(A[0], fx(F[4]), S[2], one[0]);
        S[3] = fx_mad1(A[1], fx(F[2]), S[3], one[1]);
        S[4] = fx_mad1(A[1], fx(F[6]), S[4], one[1]);
        S[5] = fx_mad1(A[1], fx(F[8]), S[5], one[1]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            S[6 + i] = fx_mad1(A[2], fx(F[3 + 2 * i]), S[6 + i], one[2]);
            S[10 + i] = fx_mad1(A[3], fx(F[3 + 2 * i]), S[10 + i], one[3]);
        }
    }
    acc[kPhi] = fma(r * m, FU, fma(-ru, Fd, acc[kPhi]));
    const double hL = (r * FL) * L, hH = (r * FH) * H;
    acc[kL0] += hL;
    acc[kL1] = fma(hL, tau, acc[kL1]);
    acc[kH0] += hH;
    acc[kH1] = fma(hH, tau, acc[kH1]);
    const double y1 = r * Y1, y2 = r * fma(Ci, FV, -(Cr * X));
    acc[kY10] += y1;
    acc[kY11] = fma(y1, tau, acc[kY11]);
    acc[kY20] += y2;
    acc[kY21] = fma(y2, tau, acc[kY21]);
    const double g = r * __longlong_as_double(bG & 0x7FFFFFFFFFFFFFFFll), gq = g * q, gt = g * tau;
    acc[kGa] = fma(g, FL, acc[kGa]);
    acc[kGb] = fma(g, FH, acc[kGb]);
    acc[kGc] = fma(gq, FV, acc[kGc]);
    acc[kGd] = fma(gq, X, acc[kGd]);
    acc[kGt1] = fma(gt, fx_to_double(fsum, pw.hexp), acc[kGt1]);              // (FL + FH) / 2
    acc[kGt2] = fma(gq * tau, FV, acc[kGt2]);
}

// NLL and gradient of one segment; lane a holds accumulator a in v, lane j writes
// component j.  Term k's share of the rate's sum, R_k = sum r f_k (its time
// function times its part of b_k), and R'_k, the same with i b_k for b_k, come
// from the 14 sums, one per lane.  With |A_i|^2 = X_i (X = (1 - F_S) x_i for the P
// wave, F_S for the S wave) every term is sqrt(X_i X_j) e^{i psi} times functions
// of other parameters: with Z_i the sum of R_k over the amplitudes i of the terms
// (twice for |A_i|^2),
//   dR/dA0sq = (Z_0 / x_0 - Z_pa / x_pa) / 2,  dR/dApesq = (Z_pe / x_pe - Z_pa / x_pa) / 2,
//   dR/dF_S = (Z_S / F_S - (Z_0 + Z_pa + Z_pe) / (1 - F_S)) / 2,
// and the phases' derivatives are sums of +-R'_k.  Then
//   dNLL/dtheta = -cs dR/dtheta + cs dlnN/dtheta SR,  SR = sum_k R_k,
//   dNLL/df_b = SR / N - Q / V.
template <bool GRAD, bool CACHED>
__device__ __forceinline__ void phis_finalize(const PhisConsts& c, double v, int n_par, double* out, int lane) {
    if (lane == 0) out[0] = -v;
    if (!GRAD) return;
    constexpr unsigned kAll = 0xffffffffu;
    auto A = [&](int i) { return __shfl_sync(kAll, v, i); };
    const double D2 = 2.0 * c.D;
    // lanes 0-9: R_k; 10-15: R'_k of k = 3, 4, 5, 7, 8, 9; 16-18: R_k / C_SP of k = 7, 8, 9
    double R;
    {
        const int pk = lane - 10;
        const int k = lane < 10 ? lane : (lane < 16 ? (pk < 3 ? 3 + pk : 4 + pk) : (lane < 19 ? lane - 9 : 0));
        const bool prime = lane >= 10 && lane < 16;
        const double re = prime ? -c.bi[k] : c.br[k], im = prime ? c.br[k] : c.bi[k];
        const double ej = kEta[kPairJ[k]];
        const bool equal = kEta[kPairI[k]] == ej;
        const int e = k == 0 ? 0 : (k == 1 ? 1 : (k == 4 ? 2 : (k == 2 ? 3 : (k == 6 ? 4 : 5))));
        const double S1 = __shfl_sync(kAll, v, equal ? kE + e : kMU + ((k - 3) >> 1));
        const double S2 = __shfl_sync(kAll, v, equal ? kE : kMV + ((k - 3) >> 1));
        const double part = kPairIm[k] ? im : re;
        const double a1 = equal ? part : (kPairIm[k] ? -ej * re : ej * im);
        const double sc = 0.25 * (lane >= 16 ? 1.0 : row_scale(c, k)) * (CACHED ? 1.0 : kBasisScale[k]);
        R = sc * (equal ? a1 * S1 : fma(a1, S1, (part * D2) * S2));
    }
    double Rk[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) Rk[k] = __shfl_sync(kAll, R, k);
    const double SR = (((Rk[0] + Rk[1]) + (Rk[2] + Rk[3])) + ((Rk[4] + Rk[5]) + (Rk[6] + Rk[7]))) + (Rk[8] + Rk[9]);
    const double csSR = c.cs * SR;
    const double p3 = __shfl_sync(kAll, R, 10), p4 = __shfl_sync(kAll, R, 11), p5 = __shfl_sync(kAll, R, 12);
    const double p7 = __shfl_sync(kAll, R, 13), p8 = __shfl_sync(kAll, R, 14), p9 = __shfl_sync(kAll, R, 15);
    const double csp = __shfl_sync(kAll, R, 16) + __shfl_sync(kAll, R, 17) + __shfl_sync(kAll, R, 18);
    const double inv = 1.0 / (lane == 0 ? c.x0 : (lane == 1 ? c.xa : (lane == 2 ? c.xe : (lane == 3 ? c.F : 1.0 - c.F))));
    const double i0 = __shfl_sync(kAll, inv, 0), ia = __shfl_sync(kAll, inv, 1), ie = __shfl_sync(kAll, inv, 2);
    const double iF = __shfl_sync(kAll, inv, 3), iP = __shfl_sync(kAll, inv, 4);
    const double Z0 = fma(2.0, Rk[0], (Rk[4] + Rk[5]) + Rk[9]), Za = fma(2.0, Rk[1], (Rk[3] + Rk[4]) + Rk[7]);
    const double Ze = fma(2.0, Rk[2], (Rk[3] + Rk[5]) + Rk[8]), ZS = fma(2.0, Rk[6], (Rk[7] + Rk[8]) + Rk[9]);
    const double Q = A(kQ), phi = A(kPhi);
    const double L0 = A(kL0), L1 = A(kL1), H0 = A(kH0), H1 = A(kH1);
    const double y10 = A(kY10);
    const double Y10 = D2 * y10, Y11 = D2 * A(kY11), Y20 = D2 * A(kY20), Y21 = D2 * A(kY21);
    const double kk = 2.0 * c.cG;
    const double ga = kk * A(kGa), gb = kk * A(kGb), gc = (kk * D2) * A(kGc), gd = (kk * D2) * A(kGd);
    const double gt = kk * fma(2.0, A(kGt1), D2 * A(kGt2));
    double d = 0.0;      // cs sum r dR/dtheta of the lane's parameter
    if (lane == IPA_GAMMA) {
        d = c.s2 * ((c.GL * L0 + c.GH * H0) + (c.Gamma * Y10 + c.Dm * Y20) - ((ga + gb) + gc)) - ((L1 + H1) + Y11);
    } else if (lane == IPA_SIGMA) {
        const double g2 = (c.Gamma - c.Dm) * (c.Gamma + c.Dm), gd2 = 2.0 * c.Gamma * c.Dm;
        d = c.sigma * ((c.GL * (c.GL * L0 - ga) + c.GH * (c.GH * H0 - gb)) + (g2 * Y10 + gd2 * Y20) -
                       (c.Gamma * gc - c.Dm * gd)) - c.inv_s * gt;
    } else if (lane == IPA_MU) {
        d = (c.GL * L0 + c.GH * H0) + (c.Gamma * Y10 + c.Dm * Y20) - ((ga + gb) + gc);
    } else if (lane == IPA_PHIS_DG) {
        d = 0.5 * (c.s2 * ((c.GL * L0 - c.GH * H0) - (ga - gb)) - (L1 - H1));
    } else if (lane == IPA_PHIS_DM) {
        d = c.s2 * ((c.Gamma * Y20 - c.Dm * Y10) + gd) - Y21;
    } else if (lane == IPA_A0SQ) {
        d = 0.5 * c.cs * (Z0 * i0 - Za * ia);
    } else if (lane == IPA_APESQ) {
        d = 0.5 * c.cs * (Ze * ie - Za * ia);
    } else if (lane == IPA_DPA) {
        d = c.cs * ((p4 + p7) - p3);
    } else if (lane == IPA_DPE) {
        d = c.cs * ((p3 + p5) + p8);
    } else if (lane == IPA_FS) {
        d = 0.5 * c.cs * (ZS * iF - ((Z0 + Za) + Ze) * iP);
    } else if (lane == IPA_DS) {
        d = c.cs * (-((p7 + p8) + p9));
    } else if (lane == IPA_PHIS_PHIS) {
        d = phi;
    } else if (lane == IPA_PHIS_OMEGA) {
        d = -4.0 * y10;
    } else if (lane == IPA_PHIS_CSP) {
        d = c.cs * (csp);
    }
    if (lane < IPA_NPAR_PHIS)
        out[1 + lane] = lane == IPA_FB ? fma(SR, c.inv_N, -Q * c.inv_V)
                        : (lane == IPA_PHIS_QNORM ? 0.0 : fma(c.dlnN[lane], csSR, -d));
    for (int j = IPA_NPAR_PHIS + lane; j < n_par; j += 32) out[1 + j] = 0.0;
}

// Three blocks per SM (168 registers, no spills) over two (200): 404 -> 367 us for
// 1e6 events, and four (128 registers, spills) 392 us; with the time functions and the
// angles in cheap fixed-point products (fast_fixed.cuh, faddeeva.cuh) 300 us.  The 40-product form with
// its 47 sums took 623 us at two blocks (237 registers).  A tile's team is the
// block's four warps (each takes 4 of every lane's 16 events), so that a small
// fit's tiles run four FP64 instruction streams at once.
template <bool GRAD, bool WEIGHTED, bool CACHED>
__global__ void __launch_bounds__(32 * kTeam, 3)
phis_kernel(Cols cols, int64_t n, const int64_t* __restrict__ seg_begin, const int64_t* __restrict__ seg_end,
            const int64_t* __restrict__ seg_tiles, int n_seg, const Consts* __restrict__ consts,
            double* __restrict__ partials, unsigned* __restrict__ counters, unsigned* __restrict__ gcount,
            unsigned* __restrict__ work, double* __restrict__ out, int n_par, int per_take) {
    constexpr int NA = GRAD ? kNA : 1;
    const int out_stride = GRAD ? 1 + n_par : 1;
    __shared__ MathTables mt;
    __shared__ int64_t s_take[2];
    __shared__ double xbuf[2][kTeam][32];
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int n_wib = kTeam;
    TagSlow* const sbuf = reinterpret_cast<TagSlow*>(dyn_smem) + wib * (kSub * 32);
    PhisWarp& pw = reinterpret_cast<PhisWarp*>(dyn_smem + (size_t)n_wib * kSub * 32 * sizeof(TagSlow))[wib];

    load_math_tables(&mt);
    __syncthreads();
    asm volatile("griddepcontrol.wait;" ::: "memory");

    const bool single = seg_begin == nullptr;
    const int64_t total = single ? (n + kTile - 1) / kTile : __ldg(seg_tiles + n_seg);
    if (blockIdx.x == 0) {
        for (int s = threadIdx.x; s < n_seg; s += blockDim.x) {
            const bool empty = single ? (n == 0) : (__ldg(seg_tiles + s + 1) == __ldg(seg_tiles + s));
            if (empty)
                for (int j = 0; j < out_stride; ++j) out[(size_t)s * out_stride + j] = 0.0;
        }
    }

    // The team (the block's four warps) takes tiles together; the next take is
    // fetched while the last tile of one is in work.  s_take and xbuf are used in
    // turns, so that one barrier per tile orders their writes after the reads of
    // the turn before.
    int cur = -1, turn = 0, par = 0;
    if (threadIdx.x == 0) s_take[0] = (int64_t)atomicAdd(work, 1u) * per_take;
    __syncthreads();
    for (;; turn ^= 1) {
        const int64_t first = s_take[turn];
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
                __syncwarp();
                const double* src = reinterpret_cast<const double*>(consts + seg);
                double* dst = reinterpret_cast<double*>(&pw.c);
                for (int i = lane; i < kPhisDoubles; i += 32) dst[i] = __ldg(src + i);
                __syncwarp();
                phis_coefficients(pw, CACHED, lane);
                __syncwarp();
                cur = seg;
            }

            double acc[NA];
#pragma unroll
            for (int a = 0; a < NA; ++a) acc[a] = 0.0;
            double prod = 1.0;
            int esum = 0;
            const int64_t tbase = ev0 + (tile - t0) * kTile;
            const unsigned below = (1u << lane) - 1u;
            // warp w of the team takes events [4 w, 4 w + 4) of each lane's 16
            {
                const int i0 = wib * kSub;
                unsigned m0, m1, m2, m3;
                {
                    unsigned mk[kSub];
#pragma unroll
                    for (int k = 0; k < kSub; ++k) {
                        const int64_t e = tbase + lane + 32 * (i0 + k);
                        const bool slow = e < ev1 && !greater(__ldg(cols.t + e), pw.c.tcut);
                        mk[k] = __ballot_sync(0xffffffffu, slow);
                    }
                    m0 = mk[0];
                    m1 = mk[1];
                    m2 = mk[2];
                    m3 = mk[3];
                }
                const int p1 = __popc(m0), p2 = p1 + __popc(m1), p3 = p2 + __popc(m2);
                const int n_slow = p3 + __popc(m3);
                for (int j = lane; j < n_slow; j += 32) {
                    const int k = (j >= p1) + (j >= p2) + (j >= p3);
                    const unsigned m = k == 0 ? m0 : (k == 1 ? m1 : (k == 2 ? m2 : m3));
                    const int before = k == 0 ? 0 : (k == 1 ? p1 : (k == 2 ? p2 : p3));
                    const int64_t e = tbase + nth_set(m, j - before) + 32 * (i0 + k);
                    sbuf[j] = tag_slow(pw.c, __ldg(cols.t + e) - pw.c.mu, &mt);
                }
                __syncwarp();
                const auto slow_of = [&](int k) {
                    const unsigned m = k == 0 ? m0 : (k == 1 ? m1 : (k == 2 ? m2 : m3));
                    const int before = k == 0 ? 0 : (k == 1 ? p1 : (k == 2 ? p2 : p3));
                    TagSlow sl = {0.0, 0.0, 0.0, 0.0, 0.0};
                    if ((m >> lane) & 1u) sl = sbuf[before + __popc(m & below)];
                    return sl;
                };
                bool plain = true;
                int top = pw.rtop;
                if (GRAD && pw.fixed && ev1 - tbase >= kFewEvents) {
                    if (WEIGHTED) {
                        // the exponent of the rows' largest |w| (0 where all weights are 1; the rows read them again)
                        unsigned hi = 0;
#pragma unroll
                        for (int k = 0; k < kSub; ++k) {
                            const int64_t e = tbase + lane + 32 * (i0 + k);
                            const double w = e < ev1 ? __ldg(cols.w + e) : 0.0;
                            hi = max(hi, (unsigned)((unsigned long long)__double_as_longlong(w) >> 32) & 0x7FFFFFFFu);
                        }
                        top += (int)(__reduce_max_sync(0xffffffffu, hi) >> 20) - 1023;
                    }
                    plain = top < -900 || top > 900;
                }
                if (!plain) {
                    long long S[14];
#pragma unroll
                    for (int a = 0; a < 14; ++a) S[a] = 0;
                    bool bad = false;
#pragma unroll 1
                    for (int k = 0; k < kSub; ++k) {
                        const int64_t e = tbase + lane + 32 * (i0 + k);
                        if (e < ev1) phis_event_fast<WEIGHTED, CACHED>(pw, &mt, cols, e, slow_of(k), top, acc, S, &prod, &esum, &bad);
                    }
                    // (none of the sums reaches 2^-4 of a typical term's 2^48 units: few of their bits would be
                    // left, as far from the peak with f_b near 1)
                    unsigned long long mag = 0;
#pragma unroll
                    for (int a = 0; a < 14; ++a) mag |= (unsigned long long)(S[a] ^ (S[a] >> 63));
                    plain = __any_sync(0xffffffffu, bad) || !__any_sync(0xffffffffu, (mag >> 44) != 0ull);
#pragma unroll
                    for (int a = 0; a < NA; ++a) {
                        if (a >= kE && a < kPhi) acc[a] = fx_to_double(S[a - kE], top + 1);
                        if (plain) acc[a] = 0.0;
                    }
                    if (plain) {
                        prod = 1.0;
                        esum = 0;
                    }
                }
#pragma unroll 1
                for (int k = 0; k < kSub; ++k) {
                    const int64_t e = tbase + lane + 32 * (i0 + k);
                    if (plain && e < ev1) {
                        const double w = WEIGHTED ? __ldg(cols.w + e) : 1.0;
                        double f[10];
                        if (CACHED) {
#pragma unroll
                            for (int kk = 0; kk < 10; ++kk) f[kk] = __ldg(cols.fk + kk * cols.fk_stride + e);
                        } else {
                            phis_basis(__ldg(cols.ck + e), __ldg(cols.cl + e), __ldg(cols.phi + e), &mt, f);
                        }
                        phis_event<GRAD, WEIGHTED>(pw, &mt, __ldg(cols.t + e), __ldg(cols.q + e), w, f, slow_of(k), acc,
                                                   &prod, &esum);
                    }
                }
                __syncwarp();
            }
            acc[0] += log_of(prod, esum, &mt);
            // each warp reduces its lanes (lane a ends with accumulator a), and warp 0
            // adds the team's four in warp order and commits the tile
            xbuf[par][wib][lane] = warp_butterfly<NA>(acc, lane);
            if (threadIdx.x == 32 * (kTeam - 1) && tile + 1 == stop)
                s_take[turn ^ 1] = (int64_t)atomicAdd(work, 1u) * per_take;
            __syncthreads();
            if (wib == 0) {
                double v = ((xbuf[par][0][lane] + xbuf[par][1][lane]) + xbuf[par][2][lane]) + xbuf[par][3][lane];
                if (row_commit<NA, GRAD ? kRow : 1>(lane, tile, t0, t1, seg, partials, gcount, counters, &v)) {
                    phis_finalize<GRAD, CACHED>(pw.c, v, n_par, out + (size_t)seg * out_stride, lane);
                    if (lane == 0) counters[seg] = 0u;
                }
            }
            par ^= 1;
        }
    }
    work_done(work, lane);
}

template <bool GRAD, bool WEIGHTED, bool CACHED>
ipa_status launch_phis_t(const Cols& cols, int64_t n, const int64_t* seg_begin, const int64_t* seg_end,
                         const int64_t* seg_tiles, int n_seg, const Consts* consts, Scratch* sc, double* out,
                         int n_par, cudaStream_t st, const LaunchCfg* force) {
    const bool single = seg_begin == nullptr;
    const int64_t tiles = tile_estimate(n, n_seg);
    if (GRAD && single && sc->partials_cap < (size_t)((n + kTile - 1) / kTile) * kRow) {
        set_error("phi_s likelihood: the scratch holds too few accumulators per tile");
        return IPA_ERR_ARG;
    }
    const LaunchCfg cfg = force ? *force : launch_cfg(IPA_MODEL_PHIS, GRAD, CACHED, n_seg > 1, tiles);
    // one block = one team of four warps sharing each tile (the geometry's
    // warps per block does not apply; its tiles per take and resident blocks do)
    const int W = kTeam;
    const int K = cfg.tiles_per_take >= 1 ? cfg.tiles_per_take : 1;
    const size_t per_warp = sizeof(PhisWarp) + kSub * 32 * sizeof(TagSlow);
    const size_t smem = (size_t)W * per_warp;
    auto kern = phis_kernel<GRAD, WEIGHTED, CACHED>;
    static bool attr[64] = {};
    static int occ[64][kMaxWarps + 1] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (!attr[dev & 63]) {
        ipa_status q = cuda_fail(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem),
                                 "phi_s kernel attribute");
        if (q != IPA_OK) return q;
        attr[dev & 63] = true;
    }
    int& per_sm = occ[dev & 63][W];
    if (per_sm == 0) {
        int v = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kern, 32 * W, smem);
        per_sm = e == cudaSuccess && v >= 1 ? v : 1;
    }
    const int64_t grid = launch_grid(cfg, W, K, per_sm, tiles, single);
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)grid);
    lc.blockDim = dim3(32u * W);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    cudaLaunchAttribute la[1];
    la[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    la[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = la;
    lc.numAttrs = 1;
    return cuda_fail(cudaLaunchKernelEx(&lc, kern, cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts,
                                        sc->partials, sc->counters, sc->gcount, sc->work, out, n_par, K),
                     "phi_s likelihood kernel launch");
}

template <bool GRAD, bool CACHED>
ipa_status launch_phis_w(const Cols& cols, int64_t n, const int64_t* seg_begin, const int64_t* seg_end,
                         const int64_t* seg_tiles, int n_seg, const Consts* consts, Scratch* sc, double* out,
                         int n_par, cudaStream_t st, const LaunchCfg* cfg) {
    if (cols.w)
        return launch_phis_t<GRAD, true, CACHED>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out,
                                                 n_par, st, cfg);
    return launch_phis_t<GRAD, false, CACHED>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, n_par,
                                              st, cfg);
}

// ---- generator (Sec. 7, Example 5: accept-reject with counter-based draws) ----

constexpr int kGenBins = 64;    // decay-time bins of the generator's envelope

// The envelope, piecewise constant in t: bin i = [e_i, e_i + w), e_i = t_lo +
// i w, w = (t_hi - t_lo) / 64, bound B_i >= rate there.  Every observed
// bilinear is at most |b_k| (gL + gH + 2 |gc|) and a convolved exponential
// g(tau; x) decreases in tau and is at most min(1, e^{-x tau + x^2 sigma^2 /
// 2}), taken at the left edge: B_i = (m(Gamma_L) + m(Gamma_H) + 2 m(Gamma))
// sum_k max|f_k| |b_k| r_k (r_k = |C_SP| for the S-P terms).
__device__ inline double phis_envelope_ang(const PhisConsts& c) {
    const double sF = 1.0 - c.F, rFs = c.rF * c.rs;
    const double mag[10] = {sF * c.x0, sF * c.xa, sF * c.xe, sF * c.ra * c.re, sF * c.r0 * c.ra, sF * c.r0 * c.re,
                            c.F, rFs * c.ra, rFs * c.re, rFs * c.r0};
    double ang = 0.0;
#pragma unroll
    for (int k = 0; k < 10; ++k) ang += cdetail::basis_max(k) * mag[k] * (k >= 7 ? fabs(c.csp) : 1.0);
    return ang;
}
__device__ inline double phis_envelope_bin(const PhisConsts& c, const ModelDev& m, double w, double ang, int i) {
    const double e = __dadd_rn(m.t_lo, __dmul_rn((double)i, w)) - c.mu;
    const double ML = fmin(1.0, exp(-c.GL * e + 0.5 * c.GL * c.GL * c.s2));
    const double MH = fmin(1.0, exp(-c.GH * e + 0.5 * c.GH * c.GH * c.s2));
    const double MG = fmin(1.0, exp(-c.Gamma * e + 0.5 * c.Gamma * c.Gamma * c.s2));
    return (ML + MH + 2.0 * MG) * ang;
}

// rate(t, Omega, q) = sum_k f_k r_k sum_j C_kj G_j, G = (gL, gH, q Re gc, q Im gc),
// with the exact convolutions (library exp, erfcx, the Faddeeva function).
__device__ double phis_rate_exact(const PhisConsts& c, const MathTables* mt, double t, double ck, double cl,
                                  double phi, double q) {
    const double tau = t - c.mu;
    double cr, ci;
    conv2_complex(c, tau, &cr, &ci);
    const double G[4] = {0.5 * conv2_real(c, tau, c.GL, c.uL0), 0.5 * conv2_real(c, tau, c.GH, c.uH0),
                         0.5 * q * cr, 0.5 * q * ci};
    double f[10];
    basis_unscaled(ck, cl, phi, mt, f);
    double r = 0.0;
    for (int k = 0; k < 10; ++k) {
        double row[4];
        c_row(k, c.br[k], c.bi[k], 1.0, c.c, c.s, 1.0, c.D, row);
        const double e = row[0] * G[0] + row[1] * G[1] + row[2] * G[2] + row[3] * G[3];
        r += kBasisScale[k] * f[k] * row_scale(c, k) * e;
    }
    return r;
}

// Signal candidate j of toy k: Philox calls (j, k, 0): u_bin, u_acc; (j, k, 1):
// ck, cl; (j, k, 2): phi, u_pos; (j, k, 3): u_q.  Its bin is the first i with
// u_bin C_64 <= C_{i+1} (C the running sums of B in order: the proposal is
// piecewise uniform with weights B_i), t = min(e_i + u_pos w, t_hi); the tag is
// the selected one (Q = +-1) or +1 for u_q <= 1/2 (the top bit of its first
// word clear), else -1; kept iff u_acc B_i < rate.  Background event i: (i, k,
// 4): t, ck; (i, k, 5): cl, phi; (i, k, 6): u_q.
//
// FP32: the ten terms' coefficients have only four distinct time functions (a
// term whose two amplitudes have the same CP eigenvalue takes T+ or T-, a mixed
// term U and V),
//   T+- = (gL + gH)/2 +- [cos phi_s (gL - gH)/2 + D sin phi_s q Im gc],
//   U = sin phi_s (gL - gH)/2 - D cos phi_s q Im gc,   V = D q Re gc,
// so rate = F+ T+ + F- T- + FU U + FV V with four angular sums of fourteen
// products.  quick() decides candidates above the resolution peak; those near
// it (about a seventh) are packed and take the FP32 erfc and Faddeeva
// function (conv32.cuh).  Every convolution carries the relative bound of
// conv32.cuh, every f_k the error ef of the 4D model's angular test (toygen.cu),
// and sum_k |b_k| r_k <= 3 sum_k max|f_k| |b_k| r_k = 3 ang: |rate32 - rate| <= ang
// (gL + gH + 2 C) (rel + 3 ef), doubled to spare.
struct PhisGen {
    static constexpr bool kQuickKeeps = true, kQuick64 = true;
    static constexpr int kBlocksPerSm = 3, kUnroll = 1, kBlockEvents = 0;
    struct Shared {
        PhisConsts c;
        MathTables mt;
        double B[kGenBins], C[kGenBins + 1];
        double t_lo, t_hi, w, total;
        Conv32 v;
        float Bf[kGenBins], Cf[kGenBins + 1], ef[kGenBins];   // B, C, e_i - mu
        Phase32 ph[kGenBins];  // the phase over each bin
        float wf, totalf, ang;
        float p[10];           // coefficient of f'_k in F+ or F- (equal eigenvalues)
        float u[4], x[4];      // coefficients of f'_3, f'_5, f'_7, f'_9 in FU and FV
        float cph, sph, D, C2;  // C2 = 2 max(1, |D|)
    };

    __device__ static void setup(Shared& S, const GenArgs& A) {
        const double* src = reinterpret_cast<const double*>(A.consts);
        double* dst = reinterpret_cast<double*>(&S.c);
        for (int i = threadIdx.x; i < kPhisDoubles; i += blockDim.x) dst[i] = src[i];
        load_math_tables(&S.mt);
        __syncthreads();
        const PhisConsts& c = S.c;
        const double span = __dsub_rn(A.m.t_hi, A.m.t_lo);
        const double w = __ddiv_rn(span, (double)kGenBins);
        if (threadIdx.x < kGenBins) {
            const int i = threadIdx.x;
            S.B[i] = phis_envelope_bin(c, A.m, w, phis_envelope_ang(c), i);
            S.Bf[i] = (float)S.B[i];
            const double e = __dadd_rn(A.m.t_lo, __dmul_rn((double)i, w)) - c.mu;
            S.ef[i] = (float)e;
            S.ph[i] = phase32_of(c.Dm, c.ph0, e, w);
        } else if (threadIdx.x == 96) {
            S.t_lo = A.m.t_lo;
            S.t_hi = A.m.t_hi;
            S.w = w;
            S.wf = (float)w;
            S.ang = (float)phis_envelope_ang(c);
            S.v = conv32_of(c, A.m.t_lo - c.mu, span);
            S.cph = (float)c.c;
            S.sph = (float)c.s;
            S.D = (float)c.D;
            S.C2 = 2.0f * fmaxf(1.0f, fabsf(S.D));
        } else if (threadIdx.x >= 128 && threadIdx.x < 138) {
            const int k = threadIdx.x - 128;
            const double sc = kBasisScale[k] * row_scale(c, k);
            const double ej = kEta[kPairJ[k]];
            S.p[k] = (float)(sc * (kPairIm[k] ? c.bi[k] : c.br[k]));
            if (kEta[kPairI[k]] != ej) {
                const int i = (k - 3) >> 1;          // 3, 5, 7, 9
                S.u[i] = (float)(sc * (kPairIm[k] ? -ej * c.br[k] : ej * c.bi[k]));
                S.x[i] = (float)(sc * (kPairIm[k] ? c.bi[k] : c.br[k]));
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            S.C[0] = 0.0;
            S.Cf[0] = 0.0f;
            for (int i = 0; i < kGenBins; ++i) {
                s = __dadd_rn(s, S.B[i]);
                S.C[i + 1] = s;
                S.Cf[i + 1] = (float)s;
            }
            S.total = s;
            S.totalf = (float)s;
        }
    }

    __device__ static bool usable(const Shared& S) {
        return isfinite(S.total) && S.total > 0.0 && isfinite(S.c.N) && S.c.N > 0.0;
    }

    // N is the integral over both tags (each drawn half of the time) or over the selected one
    __device__ static void acceptance(const GenArgs& A, float* acc) {
        __shared__ float sum;
        if (threadIdx.x == 0) sum = 0.0f;
        __syncthreads();
        const PhisConsts& c = *reinterpret_cast<const PhisConsts*>(A.consts);
        const double w = (A.m.t_hi - A.m.t_lo) / kGenBins;
        if (threadIdx.x < kGenBins)
            atomicAdd(&sum, (float)phis_envelope_bin(c, A.m, w, phis_envelope_ang(c), threadIdx.x));
        __syncthreads();
        if (threadIdx.x == 0)
            *acc = (c.qsel != 0.0 ? 1.0f : 0.5f) * (float)c.N / (8.0f * (float)cdetail::kPi * (float)w * sum);
    }

    // the first bin i with u C_64 <= C[i + 1]
    __device__ __forceinline__ static int bin_of(const Shared& S, double u) {
        const double target = __dmul_rn(u, S.total);
        int lo = 0, hi = kGenBins - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (target <= S.C[mid + 1]) hi = mid; else lo = mid + 1;
        }
        return lo;
    }
    // the same in FP32, or -1 where the uniform lies too near an edge of its bin
    // (u C_64 and C are off by less than 2.4e-7 C_64 together)
    __device__ __forceinline__ static int bin32(const Shared& S, uint32_t hi_word) {
        const float target = u32of(hi_word) * S.totalf;
        int lo = 0;
#pragma unroll
        for (int d = kGenBins / 2; d > 0; d >>= 1) lo += target > S.Cf[lo + d] ? d : 0;
        const float band = 3.0e-7f * S.totalf;
        return target - S.Cf[lo] > band && S.Cf[lo + 1] - target > band ? lo : -1;
    }
    __device__ __forceinline__ static double t_of(const Shared& S, int b, double u) {
        return fmin(__dadd_rn(__dadd_rn(S.t_lo, __dmul_rn((double)b, S.w)), __dmul_rn(u, S.w)), S.t_hi);
    }

    // F+, F-, FU, FV from the words of calls 1 and 2; returns 6 ef (infinite outside the bound's range)
    __device__ __forceinline__ static float sums32(const Shared& S, const U4& b, const U4& d, float* F) {
        const float ck = fmaf(2.0f, u32of(b.x), -1.0f), cl = fmaf(2.0f, u32of(b.z), -1.0f);
        const float cl2 = cl * cl;
        const float sk2 = fmaf(-ck, ck, 1.0f), sl2 = fmaf(-cl, cl, 1.0f);
        float sp, cp;
        sincospif(fmaf(2.0f, u32of(d.x), -1.0f), &sp, &cp);
        const float sksl2 = sk2 * sl2;
        const float rk = rsqrtf(sk2), rl = rsqrtf(sl2);
        const float q = sksl2 * (rk * rl);
        const float cp2 = cp * cp;
        const float qc = q * cl, a = qc * ck;
        F[0] = fmaf(S.p[0], ck * ck * sl2, fmaf(S.p[1], sk2 * fmaf(-sl2, cp2, 1.0f), S.p[4] * (a * cp)));
        F[1] = fmaf(S.p[2], sk2 * fmaf(sl2, cp2, cl2), fmaf(S.p[6], sl2, S.p[8] * (qc * sp)));
        const float f3 = sksl2 * (sp * cp), f5 = a * sp, f7 = qc * cp, f9 = ck * sl2;
        F[2] = fmaf(S.u[0], f3, fmaf(S.u[1], f5, fmaf(S.u[2], f7, S.u[3] * f9)));
        F[3] = fmaf(S.x[0], f3, fmaf(S.x[1], f5, fmaf(S.x[2], f7, S.x[3] * f9)));
        return sk2 >= 1.0e-5f && sl2 >= 1.0e-5f ? 6.0f * (5.0e-7f * (rk + rl) + 2.0e-6f) : INFINITY;
    }

    __device__ __forceinline__ static GenCode decide(const Shared& S, float u, int bin, const float* F, float ef6, const Time32& g,
                                                     float q) {
        const float half = 0.5f * (g.L + g.H), diff = 0.5f * (g.L - g.H);
        const float ci = q * S.D * g.Ci;
        const float mix = S.cph * diff + S.sph * ci;
        const float rate = F[0] * (half + mix) + F[1] * (half - mix) + F[2] * (S.sph * diff - S.cph * ci) +
                           F[3] * (q * S.D * g.Cr);
        const float err = S.ang * (g.L + g.H + S.C2 * g.C) * (2.0f * g.err + ef6);
        return decide32(u * S.Bf[bin], S.Bf[bin] * 1.5e-6f, rate, err);
    }

    __device__ __forceinline__ static float tag32(const Shared& S, const GenArgs& A, const GenIdx& j) {
        return (float)tag_of(S, S.c.qsel != 0.0 ? 0u : gen_draw(A, j, 3u).x);
    }
    __device__ __forceinline__ static double tag_of(const Shared& S, uint32_t hi) {
        return S.c.qsel != 0.0 ? S.c.qsel : ((hi >> 31) ? -1.0 : 1.0);
    }

    __device__ __forceinline__ static GenCode quick(const Shared& S, const GenArgs& A, const GenIdx& j) {
        const U4 a = gen_draw(A, j, 0u);
        const U4 d = gen_draw(A, j, 2u);
        const int bin = bin32(S, a.x);
        if (bin < 0) return kTest64;
        const float tau = fmaf(u32of(d.z), S.wf, S.ef[bin]);
        if (!(tau > S.v.near)) return kTest32;
        const U4 b = gen_draw(A, j, 1u);
        float F[4];
        const float ef6 = sums32(S, b, d, F);
        if (!(ef6 <= 1.0e-2f)) return kTest64;
        const Far32 f = conv32_far(S.v, tau, tau32_err(tau, S.ef[bin], S.wf));
        if (!f.ok) return kTest64;
        // what the oscillation can add at most, before its phase and the tag
        const float half = 0.5f * (f.L + f.H), diff = 0.5f * (f.L - f.H);
        const float still = F[0] * (half + S.cph * diff) + F[1] * (half - S.cph * diff) + F[2] * S.sph * diff;
        const float X = S.sph * (F[0] - F[1]) - S.cph * F[2];
        const float osc = fabsf(S.D) * f.C * (fabsf(X) + fabsf(F[3]));
        const float lhs = u32of(a.z) * S.Bf[bin];
        const float err = S.ang * (f.L + f.H + S.C2 * f.C) * (2.0f * f.err + ef6);
        if (lhs - S.Bf[bin] * 1.5e-6f > still + osc + err) return kDrop;
        return decide(S, u32of(a.z), bin, F, ef6, conv32(S.v, tau, tau32_err(tau, S.ef[bin], S.wf), phase32(S.ph[bin], d.z), S.ph[bin].ok),
                      tag32(S, A, j));
    }

    // near the peak
    __device__ __forceinline__ static GenCode test32(const Shared& S, const GenArgs& A, const GenIdx& j) {
        const U4 a = gen_draw(A, j, 0u);
        const U4 d = gen_draw(A, j, 2u);
        const int bin = bin32(S, a.x);
        const U4 b = gen_draw(A, j, 1u);
        float F[4];
        const float ef6 = sums32(S, b, d, F);
        if (bin < 0 || !(ef6 <= 1.0e-2f)) return kTest64;
        const float tau = fmaf(u32of(d.z), S.wf, S.ef[bin]);
        return decide(S, u32of(a.z), bin, F, ef6, conv32(S.v, tau, tau32_err(tau, S.ef[bin], S.wf), phase32(S.ph[bin], d.z), S.ph[bin].ok),
                      tag32(S, A, j));
    }

    __device__ __noinline__ static bool test64(const Shared& S, const GenArgs& A, const GenIdx& j) {
        const U4 a = gen_draw(A, j, 0u);
        const U4 b = gen_draw(A, j, 1u);
        const U4 d = gen_draw(A, j, 2u);
        const U4 e = gen_draw(A, j, 3u);
        const int bin = bin_of(S, u01_int(a.x, a.y));
        return __dmul_rn(u01_int(a.z, a.w), S.B[bin]) <
               phis_rate_exact(S.c, &S.mt, t_of(S, bin, u01_int(d.z, d.w)), sym_int(b.x, b.y), sym_int(b.z, b.w),
                               __dmul_rn(cdetail::kPi, sym_int(d.x, d.y)), tag_of(S, e.x));
    }

    __device__ __forceinline__ static void signal(const Shared& S, const GenArgs& A, const GenIdx& j, int64_t pos) {
        const U4 a = gen_draw(A, j, 0u);
        const U4 b = gen_draw(A, j, 1u);
        const U4 d = gen_draw(A, j, 2u);
        const U4 e = gen_draw(A, j, 3u);
        A.t[pos] = t_of(S, bin_of(S, u01_int(a.x, a.y)), u01_int(d.z, d.w));
        A.ck[pos] = sym_int(b.x, b.y);
        A.cl[pos] = sym_int(b.z, b.w);
        A.phi[pos] = __dmul_rn(cdetail::kPi, sym_int(d.x, d.y));
        A.q[pos] = tag_of(S, e.x);
    }

    __device__ __forceinline__ static void background(const Shared& S, const GenArgs& A, const GenIdx& i, int64_t pos) {
        const U4 a = gen_draw(A, i, 4u);
        const U4 b = gen_draw(A, i, 5u);
        const U4 e = gen_draw(A, i, 6u);
        A.t[pos] = __dadd_rn(S.t_lo, __dmul_rn(u01_int(a.x, a.y), __dsub_rn(S.t_hi, S.t_lo)));
        A.ck[pos] = sym_int(a.z, a.w);
        A.cl[pos] = sym_int(b.x, b.y);
        A.phi[pos] = __dmul_rn(cdetail::kPi, sym_int(b.z, b.w));
        A.q[pos] = tag_of(S, e.x);
    }

    __device__ __forceinline__ static void fill_nan(const GenArgs& A, int64_t pos) {
        A.t[pos] = A.ck[pos] = A.cl[pos] = A.phi[pos] = A.q[pos] = __longlong_as_double(0x7ff8000000000000ll);
    }
};

}  // namespace

ipa_status launch_phis_toygen(const GenArgs& a, cudaStream_t s) { return launch_generator<PhisGen>(a, s); }


namespace {
// ipa_nll_grad_combine for the phi_s model: the kernel's last reduction level
// over gathered group partials, then phis_finalize (one warp).
template <bool CACHED>
__global__ void phis_combine_kernel(const double* __restrict__ groups, int64_t n_groups,
                                    const Consts* __restrict__ consts, int n_par, double* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    if (n_groups == 0) {
        for (int j = lane; j < 1 + n_par; j += 32) out[j] = 0.0;
        return;
    }
    const double v = sum_rows<kNA, kRow>(groups, 0, n_groups, 1, lane);
    phis_finalize<true, CACHED>(*reinterpret_cast<const PhisConsts*>(consts), v, n_par, out, lane);
}
}  // namespace

ipa_status launch_phis_combine(const double* groups, int64_t n_groups, bool cached, const Consts* consts, int n_par,
                               double* out, cudaStream_t s) {
    if (cached)
        phis_combine_kernel<true><<<1, 32, 0, s>>>(groups, n_groups, consts, n_par, out);
    else
        phis_combine_kernel<false><<<1, 32, 0, s>>>(groups, n_groups, consts, n_par, out);
    return cuda_fail(cudaGetLastError(), "phi_s combine kernel launch");
}

ipa_status launch_phis_nll(const ModelDev& m, bool grad, const Cols& cols, int64_t n,
                           const int64_t* seg_begin, const int64_t* seg_end, const int64_t* seg_tiles, int n_seg,
                           const Consts* consts, Scratch* sc, double* out, cudaStream_t st, const LaunchCfg* cfg) {
    const int P = m.n_par;
    if (cols.fk)
        return grad ? launch_phis_w<true, true>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, P, st, cfg)
                    : launch_phis_w<false, true>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, P, st, cfg);
    return grad ? launch_phis_w<true, false>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, P, st, cfg)
                : launch_phis_w<false, false>(cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc, out, P, st, cfg);
}

}  // namespace ipa
