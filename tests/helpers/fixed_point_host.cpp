// The fixed-point functions of the likelihood kernels (fast_fixed.cuh, faddeeva.cuh)
// compiled for the host, from the headers that the kernels include: CUDA's
// integer intrinsics are defined here by their documentation.  Compiled with
// -fsanitize=signed-integer-overflow, whose handlers (below) count: the functions'
// intended wrap-arounds are unsigned, so an overflow of a signed number is a fault.
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <cuda_runtime.h>

static long long g_overflows = 0;
extern "C" {
void __ubsan_handle_add_overflow(void*, void*, void*) { ++g_overflows; }
void __ubsan_handle_sub_overflow(void*, void*, void*) { ++g_overflows; }
void __ubsan_handle_mul_overflow(void*, void*, void*) { ++g_overflows; }
void __ubsan_handle_negate_overflow(void*, void*) { ++g_overflows; }
long long overflows() { return g_overflows; }
}

// relative change of the reciprocal and reciprocal root's FP32 seeds (the hardware's may be a few units off)
static float g_seed = 1.0f;
extern "C" void set_seed_factor(float f) { g_seed = f; }

struct Index {
    int x;
};
static const Index threadIdx = {0}, blockDim = {1};
static inline long long __double_as_longlong(double x) {
    long long v;
    memcpy(&v, &x, 8);
    return v;
}
static inline double __longlong_as_double(long long x) {
    double v;
    memcpy(&v, &x, 8);
    return v;
}
static inline unsigned __float_as_uint(float x) {
    unsigned v;
    memcpy(&v, &x, 4);
    return v;
}
static inline float __uint_as_float(unsigned x) {
    float v;
    memcpy(&v, &x, 4);
    return v;
}
static inline int __mulhi(int a, int b) { return (int)(((long long)a * b) >> 32); }
static inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }
static inline long long __mul64hi(long long a, long long b) { return (long long)(((__int128)a * b) >> 64); }
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
static inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
static inline float __frcp_rn(float x) { return 1.0f / x * g_seed; }
static inline float rsqrtf(float x) { return 1.0f / sqrtf(x) * g_seed; }
static inline double erfcx(double x) { return x; }            // (only beyond the tested ranges)

#include "faddeeva.cuh"
#include "fast_fixed.cuh"

using namespace ipa;

static const MathTables& tables() {
    static MathTables t;
    static const bool loaded = (load_math_tables(&t), true);
    (void)loaded;
    return t;
}

extern "C" {
void exp_neg(const double* x, double* y, int64_t n) {
    for (int64_t i = 0; i < n; ++i) y[i] = fx_exp_neg(x[i], &tables());
}
// log x 2^56
void log_q56(const double* x, int64_t* y, int64_t n) {
    for (int64_t i = 0; i < n; ++i) y[i] = fx_log(x[i], &tables());
}
void erfcx_fixed(const double* x, double* y, int64_t n) {
    for (int64_t i = 0; i < n; ++i) y[i] = fx_erfcx(x[i], &tables());
}
void faddeeva_fixed(const double* z, double* w, int64_t n) {
    for (int64_t i = 0; i < n; ++i) faddeeva_uhp(z[2 * i], z[2 * i + 1], w + 2 * i, w + 2 * i + 1);
}
// the decay exponential 2 e^{-Gamma (t - mu) + c_exp} and whether it is in range
int exp_line(double Gamma, double mu, double c_exp, double t_most, const double* t, double* y, int* ok, int64_t n) {
    const FxExp s = fx_exp_setup(Gamma, mu, c_exp, t_most);
    for (int64_t i = 0; i < n && s.ok; ++i) {
        bool in = fx_in_range(t[i], s.top);
        y[i] = fx_exp(fx(fx_signed(t[i], s.top)), s, &tables(), &in);
        ok[i] = in;
    }
    return s.ok;
}
// sin and cos (Q62) of Dm (t - mu) - ph0
int phase_line(double Dm, double mu, double ph0, double t_most, const double* t, int64_t* y, int64_t n) {
    const FxExp s = fx_phase_setup(Dm, mu, ph0, t_most);
    for (int64_t i = 0; i < n && s.ok; ++i) {
        long long sn, cs;
        fx_phase(fx(fx_signed(t[i], s.top)), s, &tables(), &sn, &cs);
        y[2 * i] = sn;
        y[2 * i + 1] = cs;
    }
    return s.ok;
}
// the ten angular products (Q62) of (ck, cl, phi)
void basis(const double* a, int64_t* g, int64_t n) {
    for (int64_t i = 0; i < n; ++i) {
        long long v[10];
        fx_basis(a[3 * i], a[3 * i + 1], a[3 * i + 2], &tables(), v);
        for (int k = 0; k < 10; ++k) g[10 * i + k] = v[k];
    }
}
int angles_ok(double ck, double cl, double phi) { return fx_angles_ok(ck, cl, phi); }
double to_double(int64_t v, int e2) { return fx_to_double(v, e2); }
}
