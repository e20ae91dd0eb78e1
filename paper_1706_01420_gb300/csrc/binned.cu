// Binned workloads (Example 4, CLs, and the toolkit's generateBinned and
// Gaussian smearing): Poisson pseudo-experiments of a histogram, the smearing
// of a histogram by a Gaussian, and CL_b, CL_s+b, CL_s from toys.
//
// Poisson counts.  Bin i of toy k under hypothesis h is Poisson(lambda_i) by
// inversion of the CDF with one uniform per piece from Philox-4x32-10
// (philox.cuh): counter (i lo32, i hi32, k, 8 + 2^16 h + m/2), words 2 (m mod 2)
// and 2 (m mod 2) + 1; a mean above 400 is split into M = ceil(lambda/400)
// pieces of lambda/M (Poisson counts add).  Piece of mean nu, uniform u:
//   n = 0, p = exp(-nu), F = p;  while u > F and p > 0 and n < cap:
//   n += 1, p = (p nu) / n, F += p;   cap = floor(nu + 40 sqrt(nu) + 100).
// Every step is a correctly rounded IEEE operation (no contraction), so the
// counts are reproducible bit for bit.  The recurrence depends only on the
// bin's mean, so it runs once per bin and call into a table of thresholds
// (BinTable); a draw is then one Philox block and a few integer comparisons.
//
// CLs.  With w_i = ln(1 + s_i / b_i), X = sum_i n_i w_i (the data-dependent part
// of -2 ln Q, Q = L(s+b) / L(b)); CL_s+b = P_s+b(X <= X_obs), CL_b =
// P_b(X <= X_obs), CL_s = CL_s+b / CL_b over n_toys toys per hypothesis.  The
// counts are drawn on the fly (no histogram is stored).  X is summed in a fixed
// order: bins in order within a slice of kSlice, the slices in four interleaved
// chains; the data take the same order.
//
// A lane draws one toy's bins: the 32 toys of a warp meet a bin together, so its
// thresholds (their high words: a tie goes by the whole table) and weight come as one
// broadcast from shared memory, and the first two of Philox's ten rounds are
// computed once per bin and once per toy.  Before, a block walked one toy
// with a bin per thread: every draw fetched its own 40-byte record and two or
// three doubles of the CDF from L2 (2.4 MB of tables), and converted and
// compared in FP64, four FP64 instructions per draw on a pipe of 2 per clock and
// SM.  Now one (the FMA into X).  Bound by the 32 x 32 -> 64-bit products (15 per draw) and
// issue.  10 000 bins, 10 000 toys: 3.7 ms before, 0.81 with the ten rounds per draw and
// 64-bit thresholds, 0.72 now; the tables (a serial chain per bin, run twice and to its
// end before) 305 -> 21 us for both.
#include <math.h>

#include "ipa_internal.cuh"
#include "philox.cuh"

namespace ipa {
namespace {

constexpr double kPiece = 400.0;
constexpr int kBinBlock = 256;
constexpr int kTabBlock = 64;           // bins per block of the table kernels: a bin is a serial chain, so spread them
constexpr int kTabFixed = 32;           // thresholds per bin in the fixed part of the table
constexpr int kSlice = 64;              // bins summed by one thread of the CLs kernel
constexpr int kToyBlock = 128;          // toys per block of the CLs kernel
// Thresholds compared without a search.  10 000 bins and toys, means 0.1 / 0.5 / 2 / 5 / 20 in us: 3 of them
// 681 / 892 / 1328 / 1477 / 1698, 5 711 / 724 / 1160 / 1511 / 1731, 8 765 / 772 / 835 / 1403 / 1774, 12 843 / 852 / 863 /
// 1098 / 1827: 5 for means around one half (Example 4's), where a draw passes few.
constexpr int kFirst = 5;
constexpr uint32_t kBinnedCall = 8u;

__device__ __forceinline__ uint32_t binned_call(int hyp, int m) {
    return kBinnedCall + ((uint32_t)hyp << 16) + (uint32_t)(m >> 1);
}

// The inversion of one bin, tabulated once per call and shared by every toy:
// with nu = lambda / M, p_0 = exp(-nu), cap = floor(nu + 40 sqrt(nu) + 100), the
// recurrence p_n = (p_{n-1} nu) / n, F_n = F_{n-1} + p_n (each step correctly
// rounded) gives the CDF values F_0 <= F_1 <= ...  A draw with uniform u is the
// first n with u <= F_n, or the n where the recurrence ends (p = 0 or n = cap)
// when u exceeds them all.  u = (v + 1) 2^-53 with v the top 53 bits of the
// draw's 64-bit word, so u > F_n exactly when the word is at least
// floor(F_n 2^53) 2^11: the table holds these 64-bit integers.  It ends before
// the first F_n >= 1 (which no u exceeds: the draw is n), or past the mode where
// adding p_n no longer changes F (no later n is the first).  The counts are
// those of the sequential FP64 loop bit for bit.
struct BinTable {
    int64_t off;    // first entry in the flat threshold array
    double nu;      // mean of one piece
    int M;          // pieces (0 for a non-positive mean)
    int len;        // entries
    int stop;       // the draw when the word passes every entry; -1: where the recurrence ends (bin_end)
    int pad_;
};

struct Recurrence {
    double nu, cap, p, f;
    int n;
    __device__ explicit Recurrence(double nu_) : nu(nu_), n(0) {
        cap = floor(__dadd_rn(__dadd_rn(nu, __dmul_rn(40.0, sqrt(nu))), 100.0));
        p = exp(-nu);
        f = p;
    }
    __device__ bool more() const { return p > 0.0 && (double)n < cap; }
    __device__ void next() {
        n += 1;
        p = __ddiv_rn(__dmul_rn(p, nu), (double)n);
    }
};

// Where the recurrence ends: the draw of a word past a table that stopped
// changing (about one draw in 10^15).
__device__ __noinline__ int bin_end(double nu) {
    Recurrence r(nu);
    while (r.more()) r.next();
    return r.n;
}

// One bin's thresholds: the first `room` of them into T; t gets everything but off.
__device__ inline void bin_table(double lam, BinTable* t, unsigned long long* T, int room) {
    *t = BinTable{};
    if (!(lam > 0.0)) return;
    const double Md = ceil(lam / kPiece);
    t->M = Md < 1.0 ? 1 : (int)Md;
    t->nu = __ddiv_rn(lam, (double)t->M);
    t->stop = -1;
    Recurrence r(t->nu);
    while (true) {
        if (r.f >= 1.0) {
            t->stop = t->len;
            break;
        }
        if (t->len < room) T[t->len] = (unsigned long long)(r.f * 9007199254740992.0) << 11;   // exact product, truncated
        ++t->len;
        if (!r.more()) break;
        r.next();
        const double g = __dadd_rn(r.f, r.p);
        if (g == r.f && (double)r.n > r.nu) break;
        r.f = g;
    }
}

// The first entry at or after j (all before it passed by `word`) that the word
// does not pass; t.len if it passes all.
__device__ __forceinline__ int bin_search(const BinTable& t, const unsigned long long* __restrict__ T,
                                          unsigned long long word, int j) {
    int lo = j, hi = t.len;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (word >= __ldg(T + t.off + mid)) lo = mid + 1; else hi = mid;
    }
    return lo;
}
__device__ __forceinline__ int bin_draw(const BinTable& t, const unsigned long long* __restrict__ T,
                                        unsigned long long word, int j) {
    const int n = bin_search(t, T, word, j);
    return n < t.len ? n : (t.stop >= 0 ? t.stop : bin_end(t.nu));
}

__device__ __forceinline__ unsigned long long word64(uint32_t a, uint32_t b) {
    return ((unsigned long long)a << 32) | b;
}

__device__ __forceinline__ int poisson_bin(const BinTable& t, const unsigned long long* __restrict__ T, uint64_t i,
                                           uint32_t toy, int hyp, uint32_t k0, uint32_t k1) {
    int n = 0;
    for (int m = 0; m < t.M; ++m) {
        const U4 r = draw(i, toy, binned_call(hyp, m), k0, k1);
        n += bin_draw(t, T, (m & 1) ? word64(r.z, r.w) : word64(r.x, r.y), 0);
    }
    return n;
}

// Tables of n_tab histograms over the same bins (table h: means lam, plus add
// for h = 1).  Bin x = h n_bins + i has `fixed` entries at x fixed; a longer
// table goes to the part behind them, whose entries *more counts.
__global__ void __launch_bounds__(kTabBlock)
table_kernel(const double* __restrict__ lam, const double* __restrict__ add, int64_t n_bins, int n_tab, int fixed,
             BinTable* __restrict__ tab, unsigned long long* __restrict__ T, unsigned long long* __restrict__ more) {
    const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x >= n_bins * n_tab) return;
    const int64_t i = x < n_bins ? x : x - n_bins;
    const double l = x < n_bins ? __ldg(lam + i) : __ldg(lam + i) + __ldg(add + i);
    BinTable t;
    bin_table(l, &t, T + x * fixed, fixed);
    t.off = x * fixed;
    if (t.len > fixed) t.off = -1 - (int64_t)atomicAdd(more, (unsigned long long)t.len);
    tab[x] = t;
}

// The long tables (off = -1 - place) into the second part, from entry `first` on.
__global__ void __launch_bounds__(kTabBlock)
table_long_kernel(const double* __restrict__ lam, const double* __restrict__ add, int64_t n_bins, int n_tab,
                  BinTable* __restrict__ tab, unsigned long long* __restrict__ L) {
    const int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (x >= n_bins * n_tab || tab[x].off >= 0) return;
    const int64_t i = x < n_bins ? x : x - n_bins;
    const double l = x < n_bins ? __ldg(lam + i) : __ldg(lam + i) + __ldg(add + i);
    const int64_t place = -1 - tab[x].off;
    BinTable t;
    bin_table(l, &t, L + place, tab[x].len);
}

__global__ void __launch_bounds__(kBinBlock)
generate_kernel(const BinTable* __restrict__ tab, const unsigned long long* __restrict__ T,
                const unsigned long long* __restrict__ L, int64_t n_bins, uint32_t k0, uint32_t k1, int hyp, int toy0,
                int n_toys, int32_t* __restrict__ counts) {
    const int64_t total = n_bins * (int64_t)n_toys;
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = x / n_bins, i = x - k * n_bins;
        BinTable t = tab[i];
        const unsigned long long* F = t.off >= 0 ? T : L;
        if (t.off < 0) t.off = -1 - t.off;
        counts[x] = poisson_bin(t, F, (uint64_t)i, (uint32_t)(toy0 + k), hyp, k0, k1);
    }
}

// Discrete Gaussian kernel K_d (|d| <= R), normalised to unit sum (one block).
__global__ void smear_weights_kernel(int R, double width, double sigma, double* __restrict__ K) {
    __shared__ double part[kBinBlock];
    const int n = 2 * R + 1;
    const double c = 1.0 / (2.0 * sigma * sigma);
    double acc = 0.0;
    for (int d = threadIdx.x; d < n; d += blockDim.x) {
        const double x = (d - R) * width;
        const double v = exp(-(x * x) * c);
        K[d] = v;
        acc += v;
    }
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) part[threadIdx.x] += part[threadIdx.x + s];
        __syncthreads();
    }
    const double inv = 1.0 / part[0];
    for (int d = threadIdx.x; d < n; d += blockDim.x) K[d] *= inv;
}

// out_i = sum_{|d| <= R} K_d h_{i-d}, bins outside the histogram contributing nothing.
__global__ void __launch_bounds__(kBinBlock)
smear_kernel(const double* __restrict__ h, int64_t n_bins, int R, const double* __restrict__ K,
             double* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_bins; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j0 = i - R < 0 ? 0 : i - R;
        const int64_t j1 = i + R >= n_bins ? n_bins - 1 : i + R;
        double acc = 0.0;
        for (int64_t j = j0; j <= j1; ++j) acc = fma(__ldg(K + (i - j + R)), __ldg(h + j), acc);
        out[i] = acc;
    }
}

// w_i = ln(1 + s_i / b_i).
__global__ void cls_weights_kernel(const double* __restrict__ s, const double* __restrict__ b, int64_t n_bins,
                                   double* __restrict__ w) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_bins; i += (int64_t)gridDim.x * blockDim.x)
        w[i] = log1p(__ldg(s + i) / __ldg(b + i));
}

// One bin of a slice in shared memory: the high words of its first thresholds (~0 beyond the
// table) behind a zero, its part of the draw's first rounds, its weight.
struct __align__(16) SliceBin {
    uint32_t hi[1 + kFirst];
    PhiloxRow row;
    double w;
    int first;        // min(kFirst, len): a word that passes this many needs the whole table
    int one;          // 1: one piece, 0: the general path
};
static_assert(sizeof(SliceBin) % 16 == 0, "16-byte loads");

// Slice sums of X: part[s * stride + c] = sum over the slice's bins of n_i w_i
// for column c of the batch: toy toy0 + c of hypothesis 0 (c < n) or toy toy0 +
// c - n of hypothesis 1; column 2 n, the data, if it is given (block.y = 2).
__global__ void __launch_bounds__(kToyBlock)
cls_slices_kernel(const BinTable* __restrict__ tab, const unsigned long long* __restrict__ T,
                  const unsigned long long* __restrict__ L, const double* __restrict__ w, int64_t n_bins, int64_t n_slices,
                  const __grid_constant__ PhiloxKeys keys, int toy0, int n, const int32_t* __restrict__ data,
                  double* __restrict__ part, int64_t stride) {
    __shared__ SliceBin bins[kSlice];
    __shared__ double num[kFirst + 1];
    const int hyp = blockIdx.y;
    if (hyp == 2) {                      // the data: a thread per slice
        for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n_slices; s += (int64_t)gridDim.x * blockDim.x) {
            double acc = 0.0;
            const int64_t e = (s + 1) * kSlice < n_bins ? (s + 1) * kSlice : n_bins;
            for (int64_t i = s * kSlice; i < e; ++i) {
                const int k = __ldg(data + i);
                if (k) acc = fma((double)k, __ldg(w + i), acc);
            }
            part[s * stride + 2 * n] = acc;
        }
        return;
    }
    const int64_t toy_blocks = (n + kToyBlock - 1) / kToyBlock;
    const int64_t s = blockIdx.x / toy_blocks;
    if (s >= n_slices) return;           // (block row 2 may be longer)
    const int c = (int)(blockIdx.x - s * toy_blocks) * kToyBlock + threadIdx.x;
    const int64_t i0 = s * kSlice;
    const int nb = (int)(n_bins - i0 < kSlice ? n_bins - i0 : kSlice);
    tab += (int64_t)hyp * n_bins + i0;
    if (threadIdx.x <= kFirst) num[threadIdx.x] = (double)threadIdx.x;
    for (int b = threadIdx.x; b < nb; b += kToyBlock) {
        const BinTable t = tab[b];
        SliceBin r;
        const unsigned long long* F = t.off >= 0 ? T + t.off : L + (-1 - t.off);
        r.hi[0] = 0u;
#pragma unroll
        for (int q = 0; q < kFirst; ++q) r.hi[1 + q] = q < t.len ? (uint32_t)(__ldg(F + q) >> 32) : ~0u;
        r.row = philox_row(keys, (uint32_t)(i0 + b), binned_call(hyp, 0));
        r.w = __ldg(w + i0 + b);
        r.one = t.M == 1;
        r.first = t.len < kFirst ? t.len : kFirst;
        bins[b] = r;
    }
    __syncthreads();
    if (c >= n) return;
    const uint32_t toy = (uint32_t)(toy0 + c);
    const PhiloxCol col = philox_col(keys, (uint32_t)(i0 >> 32), toy);       // (a slice has one high word)
    double acc = 0.0;
#pragma unroll 2
    for (int b = 0; b < nb; ++b) {
        const SliceBin& r = bins[b];
        if (r.one) {
            const U4 x = keyed_from<2>(keys, U4{r.row.a ^ col.y, r.row.b, r.row.c ^ col.h, col.w});
            // thresholds passed by the high word; a tie with the last one (2^-32) and a word past
            // them all go by the whole table
            int k = 0;
#pragma unroll
            for (int q = 1; q <= kFirst; ++q) k += x.x >= r.hi[q];
            double m = num[k];
            if (k >= r.first || x.x == r.hi[k]) {
                BinTable t = tab[b];
                const unsigned long long* F = t.off >= 0 ? T : L;
                if (t.off < 0) t.off = -1 - t.off;
                k = bin_draw(t, F, word64(x.x, x.y), 0);
                m = (double)k;
            }
            if (k) acc = fma(m, r.w, acc);           // (an infinite w counts only where there are events)
        } else {
            BinTable t = tab[b];
            const unsigned long long* F = t.off >= 0 ? T : L;
            if (t.off < 0) t.off = -1 - t.off;
            const int k = poisson_bin(t, F, (uint64_t)(i0 + b), toy, hyp, keys.k[0], keys.k[1]);
            if (k) acc = fma((double)k, r.w, acc);
        }
    }
    part[s * stride + (int64_t)hyp * n + c] = acc;
}

// X of a column from its slice sums: four interleaved chains.
__device__ __forceinline__ double sum_slices(const double* __restrict__ part, int64_t n_slices, int64_t stride) {
    double a[4] = {0.0, 0.0, 0.0, 0.0};
    int64_t s = 0;
    for (; s + 16 <= n_slices; s += 16) {            // sixteen loads in flight
        double x[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) x[q] = __ldg(part + (s + q) * stride);
#pragma unroll
        for (int q = 0; q < 16; ++q) a[q & 3] += x[q];
    }
    for (; s + 4 <= n_slices; s += 4) {
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] += __ldg(part + (s + q) * stride);
    }
    for (int q = 0; s + q < n_slices; ++q) a[q] += __ldg(part + (s + q) * stride);
    return (a[0] + a[1]) + (a[2] + a[3]);
}

// X_obs from the data's slice sums (column 2 n of a batch's partials; one thread).
__global__ void cls_obs_kernel(const double* __restrict__ part, int64_t n_slices, int64_t stride, double* __restrict__ x_obs) {
    *x_obs = sum_slices(part, n_slices, stride);
}

// X of the batch's toys, and the counts of X <= X_obs per hypothesis.
__global__ void __launch_bounds__(kBinBlock)
cls_sum_kernel(const double* __restrict__ part, int64_t n_slices, int64_t stride, int n, const double* __restrict__ x_obs,
               double* __restrict__ xb, double* __restrict__ xsb, unsigned long long* __restrict__ cnt) {
    const double xo = *x_obs;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool in = c < 2 * (int64_t)n, sb = c >= n;
    double X = 0.0;
    if (in) {
        X = sum_slices(part + c, n_slices, stride);
        if (xb) (sb ? xsb + (c - n) : xb + c)[0] = X;
    }
    const unsigned mb = __ballot_sync(0xffffffffu, in && !sb && X <= xo);
    const unsigned ms = __ballot_sync(0xffffffffu, in && sb && X <= xo);
    if ((threadIdx.x & 31) == 0) {
        if (mb) atomicAdd(cnt, (unsigned long long)__popc(mb));
        if (ms) atomicAdd(cnt + 1, (unsigned long long)__popc(ms));
    }
}

__global__ void cls_final_kernel(const unsigned long long* __restrict__ cnt, int n_toys, double* __restrict__ cl,
                                 int64_t* __restrict__ counts) {
    const double nb = (double)cnt[0], nsb = (double)cnt[1];
    const double clb = nb / n_toys, clsb = nsb / n_toys;
    cl[0] = clb;
    cl[1] = clsb;
    cl[2] = cnt[0] ? clsb / clb : __longlong_as_double(0x7ff8000000000000ll);
    if (counts) {
        counts[0] = (int64_t)cnt[0];
        counts[1] = (int64_t)cnt[1];
    }
}

int grid_for(int64_t work) {
    const int64_t g = (work + kBinBlock - 1) / kBinBlock;
    const int64_t cap = (int64_t)sm_count() * 16;
    return (int)(g < 1 ? 1 : (g > cap ? cap : g));
}

// The tables of one histogram (add == nullptr) or of lam and lam + add, in
// stream-ordered memory.  Synchronises the stream once (the size of the second
// part; nothing of it is needed where every table fits kTabFixed entries), twice where memory is short.
struct Tables {
    BinTable* tab = nullptr;
    unsigned long long *T = nullptr, *L = nullptr, *more = nullptr;
    cudaStream_t s;
    explicit Tables(cudaStream_t s_) : s(s_) {}
    ~Tables() { release(); }
    void release() {
        pool_free(tab, s);
        pool_free(T, s);
        pool_free(L, s);
        tab = nullptr;
        T = L = more = nullptr;
    }
    // Memory for n x kTabFixed entries (256 bytes a bin) may be refused where the tables themselves
    // would fit: then every table goes to the second part, of just their size.
    ipa_status build(const double* lam, const double* add, int64_t n_bins) {
        ipa_status st = build_with(kTabFixed, lam, add, n_bins);
        if (st != IPA_ERR_OOM) return st;
        cudaGetLastError();
        release();
        return build_with(0, lam, add, n_bins);
    }
    ipa_status build_with(int fixed, const double* lam, const double* add, int64_t n_bins) {
        const int n_tab = add ? 2 : 1;
        const size_t n = (size_t)n_bins * n_tab;
        ipa_status st = pool_alloc((void**)&tab, sizeof(BinTable) * n, s, "binned tables");
        if (st == IPA_OK) st = pool_alloc((void**)&T, 8 * (n * fixed + 1), s, "binned tables");
        if (st != IPA_OK) return st;
        more = T + n * fixed;
        if ((st = cuda_fail(cudaMemsetAsync(more, 0, 8, s), "binned table size")) != IPA_OK) return st;
        const unsigned grid = (unsigned)((n + kTabBlock - 1) / kTabBlock);
        table_kernel<<<grid, kTabBlock, 0, s>>>(lam, add, n_bins, n_tab, fixed, tab, T, more);
        unsigned long long h = 0;
        if ((st = cuda_fail(cudaMemcpyAsync(&h, more, 8, cudaMemcpyDeviceToHost, s), "binned table size")) != IPA_OK)
            return st;
        if ((st = cuda_fail(cudaStreamSynchronize(s), "binned table size")) != IPA_OK) return st;
        if (h) {
            if ((st = pool_alloc((void**)&L, 8 * (size_t)h, s, "binned tables")) != IPA_OK) return st;
            table_long_kernel<<<grid, kTabBlock, 0, s>>>(lam, add, n_bins, n_tab, tab, L);
        }
        return cuda_fail(cudaGetLastError(), "binned table launch");
    }
};

}  // namespace
}  // namespace ipa

extern "C" ipa_status ipa_binned_generate(const double* lambda_dev, int64_t n_bins, uint64_t seed, int32_t hypothesis,
                                          int32_t toy0, int32_t n_toys, int32_t* counts_out_dev, void* stream) {
    using namespace ipa;
    if (n_bins < 0 || n_toys < 0 || toy0 < 0 || hypothesis < 0 || hypothesis > 1 ||
        (n_bins > 0 && n_toys > 0 && (!lambda_dev || !counts_out_dev))) {
        set_error("ipa_binned_generate: bad arguments");
        return IPA_ERR_ARG;
    }
    if (n_bins == 0 || n_toys == 0) return IPA_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Tables t(s);
    ipa_status st = t.build(lambda_dev, nullptr, n_bins);
    if (st != IPA_OK) return st;
    generate_kernel<<<grid_for(n_bins * n_toys), kBinBlock, 0, s>>>(t.tab, t.T, t.L, n_bins, (uint32_t)seed,
                                                                    (uint32_t)(seed >> 32), hypothesis, toy0, n_toys,
                                                                    counts_out_dev);
    return cuda_fail(cudaGetLastError(), "binned generator launch");
}

extern "C" ipa_status ipa_binned_smear(const double* hist_dev, int64_t n_bins, double bin_width, double sigma,
                                       double* out_dev, void* stream) {
    using namespace ipa;
    if (n_bins < 0 || !(bin_width > 0.0) || !(sigma > 0.0) || (n_bins > 0 && (!hist_dev || !out_dev)) ||
        hist_dev == out_dev) {
        set_error("ipa_binned_smear: bad arguments (positive width and sigma, distinct arrays)");
        return IPA_ERR_ARG;
    }
    const double Rd = ceil(8.0 * sigma / bin_width);
    if (!(Rd <= 1e7)) {
        set_error("ipa_binned_smear: sigma spans more than 1e7 / 8 bins");
        return IPA_ERR_ARG;
    }
    if (n_bins == 0) return IPA_OK;
    const int R = (int)Rd;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    double* K = nullptr;
    ipa_status st = cuda_fail(cudaMallocAsync(&K, sizeof(double) * (2 * (size_t)R + 1), s), "smearing kernel alloc");
    if (st != IPA_OK) return st;
    smear_weights_kernel<<<1, kBinBlock, 0, s>>>(R, bin_width, sigma, K);
    smear_kernel<<<grid_for(n_bins), kBinBlock, 0, s>>>(hist_dev, n_bins, R, K, out_dev);
    st = cuda_fail(cudaGetLastError(), "smearing launch");
    cudaFreeAsync(K, s);
    return st;
}

extern "C" ipa_status ipa_cls(const double* s_dev, const double* b_dev, int64_t n_bins, const int32_t* data_dev,
                              int32_t n_toys, uint64_t seed, double* cl_out_dev, int64_t* counts_out_dev,
                              double* x_out_dev, void* stream) {
    using namespace ipa;
    if (n_bins < 1 || n_toys < 1 || !s_dev || !b_dev || !data_dev || !cl_out_dev) {
        set_error("ipa_cls: bad arguments");
        return IPA_ERR_ARG;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    Tables t(s);
    ipa_status st = t.build(b_dev, s_dev, n_bins);
    if (st != IPA_OK) return st;
    // the toys go in batches whose slice sums take at most kPartBytes
    constexpr size_t kPartBytes = 48u << 20;
    const int64_t n_slices = (n_bins + kSlice - 1) / kSlice;
    int64_t batch = (int64_t)(kPartBytes / (2 * sizeof(double)) / (size_t)n_slices) / kToyBlock * kToyBlock;
    if (batch < kToyBlock) batch = kToyBlock;
    if (batch > n_toys) batch = n_toys;
    const int64_t stride = 2 * batch + 1;
    // two counters, X_obs, w per bin, the slice sums
    const size_t bytes = 32 + sizeof(double) * ((size_t)n_bins + (size_t)(n_slices * stride));
    unsigned char* buf = nullptr;
    if ((st = pool_alloc((void**)&buf, bytes, s, "cls scratch")) != IPA_OK) return st;
    unsigned long long* cnt = reinterpret_cast<unsigned long long*>(buf);
    double* obs = x_out_dev ? x_out_dev + 2 * (size_t)n_toys : reinterpret_cast<double*>(buf + 16);
    double* w = reinterpret_cast<double*>(buf + 32);
    double* part = w + n_bins;
    PhiloxKeys keys(seed);
    cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned long long), s);
    cls_weights_kernel<<<grid_for(n_bins), kBinBlock, 0, s>>>(s_dev, b_dev, n_bins, w);
    const int64_t data_blocks = (n_slices + kToyBlock - 1) / kToyBlock;
    for (int64_t k = 0; k < n_toys; k += batch) {
        const int n = (int)(n_toys - k < batch ? n_toys - k : batch);
        const int64_t blocks = n_slices * ((n + kToyBlock - 1) / kToyBlock);
        const int64_t x = k == 0 && data_blocks > blocks ? data_blocks : blocks;
        cls_slices_kernel<<<dim3((unsigned)x, k == 0 ? 3 : 2), kToyBlock, 0, s>>>(
            t.tab, t.T, t.L, w, n_bins, n_slices, keys, (int)k, n, data_dev, part, stride);
        if (k == 0) cls_obs_kernel<<<1, 1, 0, s>>>(part + 2 * n, n_slices, stride, obs);
        cls_sum_kernel<<<(unsigned)((2 * (int64_t)n + kBinBlock - 1) / kBinBlock), kBinBlock, 0, s>>>(
            part, n_slices, stride, n, obs, x_out_dev ? x_out_dev + k : nullptr,
            x_out_dev ? x_out_dev + n_toys + k : nullptr, cnt);
    }
    cls_final_kernel<<<1, 1, 0, s>>>(cnt, n_toys, cl_out_dev, counts_out_dev);
    st = cuda_fail(cudaGetLastError(), "cls launch");
    pool_free(buf, s);
    return st;
}
