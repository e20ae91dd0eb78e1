// A tile's fixed-point sums, by one warp or by a team of four (nll.cu, tagged.cu).
//
// Rows of 32 events are taken kSub at a time (a quarter of a tile).  A quarter's
// FP64 sums start from zero and are added to the tile's in quarter order; the
// fixed-point ones are exact.  So a tile has the same bits whether one warp takes
// its four quarters in turn (solo_tile) or the four warps of a block take one each
// (team_kernel).  If the tile cannot take the fixed-point path, its quarters are
// redone by the plain loop in the same order.
//
// Which one: a team spreads a tile over the SM's four sub-partitions, each with its
// own FP64 unit, and a small call over four times as many warps; a warp of its own
// needs no exchange between warps.  launch_team_ok has the line between them.
//
// A model is a struct M with
//   Record, Slow (a near-peak event's values), kSums: FP64 sums, kInts: integer sums, NA;
//   usable(c, events, &sc)                      the scales at unit weight, false: plain loop;
//   kTopRange                                   |sc.top| beyond it: plain loop;
//   kPlainBelow                                 segments of fewer events never use the integers;
//   kLeast                                      no factor of the tile reaches 2^(top - kLeast): plain loop;
//   quarter<W>(c, mt, cols, tbase, i0, ev1, sbuf, wbuf, lane, sc, s);   (wbuf: the lane's weights)
//   bad(c, sc, s)                               a value left its range;
//   accumulators(c, sc, s, acc);
//   plain<W>(c, mt, cols, i0, i1, tbase, ev1, sbuf, lane, acc, &prod, &esum);
//   finish(c, acc, n_par, out, lane).
#pragma once

#include "fast_fixed.cuh"
#include "ipa_internal.cuh"
#include "tile_reduce.cuh"

namespace ipa {

constexpr int kSub = 4;                              // rows per quarter
constexpr int kPerLane = kTile / 32;                 // events per lane per tile
constexpr int kTeam = kPerLane / kSub;               // warps that share a tile
static_assert(kSub == 4 && kPerLane % kSub == 0, "a quarter keeps four ballot masks");

// The angular sums' unit is 2^-48 of a typical term, which a handful of events with small
// angular products would show: a tile of fewer events takes the plain loop.
constexpr int kFewEvents = 64;

// The scales of a tile's integers: its factors, and tau in the Gaussian's sums.
struct FastScale {
    int top, gtop;
};

// A lane's sums over rows on the fixed-point path: FP64 ones, the product of the P's of
// events without weight (mantissas, exponents), integers, and the high words of the
// largest factor, of the largest |tau| (gtau_most: of those that enter the Gaussian's sums)
// and of the least and largest P.
template <int NF, int NG>
struct FastSums {
    double f[NF];
    double prod;
    long long g[NG];
    int esum;
    int most, tau_most, gtau_most, p_least, p_most;
};

template <int NF, int NG>
__device__ __forceinline__ void clear(FastSums<NF, NG>& s) {
#pragma unroll
    for (int i = 0; i < NF; ++i) s.f[i] = 0.0;
    s.prod = 1.0;
#pragma unroll
    for (int i = 0; i < NG; ++i) s.g[i] = 0;
    s.esum = 0;
    s.most = s.tau_most = s.gtau_most = 0;
    s.p_least = s.p_most = 0x3FF00000;               // 1.0
}

// Sums over a lane's 16 events of factors below 2^(top - 6), in units of 2^(top - 63), and of
// their products with tau at `ttop`, |tau| < 1.75 2^(ttop - 1): a product (the factor shifted up
// by 3) is below 1.75 2^58, the sum below 1.75 2^62.  `most` and `tau` are high words.
__device__ __forceinline__ bool beyond_factor(int most, int top) { return (most >> 20) > 1023 - 7 + top; }
__device__ __forceinline__ bool beyond_tau(int tau, int ttop) { return tau >= ((1022 + ttop) << 20 | 0xC0000); }

// P outside [2^-125, 2^126) (the Newton reciprocal's range) or not a number in some event.
template <int NF, int NG>
__device__ __forceinline__ bool p_out_of_range(const FastSums<NF, NG>& s) {
    return s.p_least < 0x38200000 || s.p_most >= 0x47D00000;
}
template <int NF, int NG>
__device__ __forceinline__ void note_p(double P, FastSums<NF, NG>& s) {
    const int h = (int)(__double_as_longlong(P) >> 32);   // negative for P < 0
    s.p_least = min(s.p_least, h);
    s.p_most = max(s.p_most, h);
}

// The log term of an event: w log P, or P into the lane's product for weight 1.
template <bool WEIGHTED, class S>
__device__ __forceinline__ void add_log(double P, double w, const MathTables* mt, double* sum, S& s) {
    note_p(P, s);
    if (WEIGHTED) {
        const bool one = __double_as_longlong(w) == 0x3FF0000000000000ll;
        *sum = fma(one ? 0.0 : w, fx_to_double(fx_log(P, mt), 6), *sum);
        log_mul_nb(one ? P : 1.0, &s.prod, &s.esum);
    } else {
        log_mul_nb(P, &s.prod, &s.esum);
    }
}

// The exponent of the largest |w| of a quarter (0 where all weights are 1, as without
// weights; -1023 for subnormal ones), or kNoWeight where all are zero.  The lane keeps its
// weights in wbuf for the quarter: a second read of the column would go over the host link again
// where it lies in host memory (8e6 weighted 4D events there: read twice per tile 2.14 ms, twice
// per quarter 1.95, once 1.74).  ONCE: nothing reads these weights again, so they leave the L1
// cache to the times, which are read twice (1e6 1D events in host memory 119 -> 115 us; a team's
// warps read the quarters before their own as well).
constexpr int kNoWeight = -5000;
template <bool ONCE>
__device__ __forceinline__ double load_weight(const double* p) {
    if (!ONCE) return __ldg(p);
    double w;
    asm volatile("ld.global.nc.L1::no_allocate.f64 %0, [%1];" : "=d"(w) : "l"(p));
    return w;
}
template <bool ONCE>
__device__ __forceinline__ int weight_exponent(const Cols& cols, int64_t tbase, int i0, int64_t ev1, double* wbuf,
                                               int lane) {
    int hi = 0;
#pragma unroll
    for (int i = 0; i < kSub; ++i) {
        const int64_t e = tbase + lane + 32 * (i0 + i);
        const double w = e < ev1 ? load_weight<ONCE>(cols.w + e) : 0.0;
        wbuf[i * 32 + lane] = w;
        hi = max(hi, high_word(w) | (int)((unsigned)__double_as_longlong(w) != 0u));   // not 0 for any w but 0
    }
    const unsigned most = __reduce_max_sync(0xffffffffu, (unsigned)hi);
    return most ? (int)(most >> 20) - 1023 : kNoWeight;
}

// A weighted quarter's scale follows the largest |w| of its tile up to it (run); the sums
// of the quarters before, at a lower scale, are shifted to it.
template <int NF, int NG>
__device__ __forceinline__ void raise_scale(FastSums<NF, NG>& s, int run, int next) {
    if (run == kNoWeight || next <= run) return;
    const int d = next - run > 63 ? 63 : next - run;
#pragma unroll
    for (int i = 0; i < NG; ++i) s.g[i] >>= d;
}
template <class M>
__device__ __forceinline__ bool scale_to(FastScale* sc, int base, int run) {
    sc->top = base + (run == kNoWeight ? 0 : run);
    return sc->top >= -M::kTopRange && sc->top <= M::kTopRange;
}

// The integers' unit is set for typical factors.  A tile whose largest factor lies far below
// (every signal term small beside the background, as far from the peak with f_b near 1) would
// keep few of its bits: below 2^-3 to 2^-4 of a typical one the FP64 loop adds it.  `most`: the
// tile's largest factor (high word); not asked where all weights are zero, which the integers
// hold exactly.
template <class M>
__device__ __forceinline__ bool too_small(int most, FastScale sc, int run) {
    return run != kNoWeight && most < (1023 + sc.top - M::kLeast) << 20;
}

// Rows of a tile with events below ev1, up to a whole quarter.
__device__ __forceinline__ int tile_rows(int64_t tbase, int64_t ev1) {
    const int64_t rows = (ev1 - tbase + 31) >> 5;
    return rows >= kPerLane ? kPerLane : (int)((rows + kSub - 1) / kSub) * kSub;
}

// The near-peak events (t <= tcut) of a quarter: listed by a ballot per row and evaluated
// packed, 32 per pass, into sbuf, so the FP64 pipe does not run the long branch for lanes
// that discard it.  slow(i): event i's values.
struct SlowRows {
    unsigned m[kSub];
    int p[kSub];
    // position of row q's event of this lane in sbuf, or -1
    __device__ __forceinline__ int at(int q, unsigned below, int lane) const {
        const unsigned mq = q == 0 ? m[0] : (q == 1 ? m[1] : (q == 2 ? m[2] : m[3]));
        const int before = q == 0 ? 0 : (q == 1 ? p[1] : (q == 2 ? p[2] : p[3]));
        return (mq >> lane) & 1u ? before + __popc(mq & below) : -1;
    }
};
template <class Slow, class F>
__device__ __forceinline__ void slow_rows(SlowRows& r, const Cols& cols, double tcut, int64_t tbase, int i0, int64_t ev1,
                                          Slow* sbuf, int lane, F slow) {
#pragma unroll
    for (int q = 0; q < kSub; ++q) {
        const int64_t e = tbase + lane + 32 * (i0 + q);
        r.m[q] = __ballot_sync(0xffffffffu, e < ev1 && !greater(__ldg(cols.t + e), tcut));
    }
    r.p[0] = 0;
    r.p[1] = __popc(r.m[0]);
    r.p[2] = r.p[1] + __popc(r.m[1]);
    r.p[3] = r.p[2] + __popc(r.m[2]);
    const int n_slow = r.p[3] + __popc(r.m[3]);
    for (int j = lane; j < n_slow; j += 32) {
        const int q = (j >= r.p[1]) + (j >= r.p[2]) + (j >= r.p[3]);
        const unsigned mq = q == 0 ? r.m[0] : (q == 1 ? r.m[1] : (q == 2 ? r.m[2] : r.m[3]));
        const int before = q == 0 ? 0 : (q == 1 ? r.p[1] : (q == 2 ? r.p[2] : r.p[3]));
        sbuf[j] = slow(tbase + nth_set(mq, j - before) + 32 * (i0 + q));
    }
    __syncwarp();
}

// Quarters [i0, i1) by the plain loop (rare): the lane's sums, product and exponent sum in
// the first NA, next and last word of `out`.
template <class M, bool W>
__device__ __noinline__ void plain_quarters(const typename M::Record& c, const MathTables* mt, const Cols& cols, int i0,
                                            int i1, int64_t tbase, int64_t ev1, typename M::Slow* sbuf, int lane,
                                            double* out) {
    double prod = 1.0;
    int esum = 0;
#pragma unroll
    for (int a = 0; a < M::NA; ++a) out[a] = 0.0;
#pragma unroll 1
    for (; i0 < i1 && tbase + 32 * i0 < ev1; i0 += kSub) {
        double q[M::NA], qp = 1.0;
#pragma unroll
        for (int a = 0; a < M::NA; ++a) q[a] = 0.0;
        M::template plain<W>(c, mt, cols, i0, i0 + kSub, tbase, ev1, sbuf, lane, q, &qp, &esum);
#pragma unroll
        for (int a = 0; a < M::NA; ++a) out[a] += q[a];
        prod *= qp;
    }
    out[M::NA] = prod;
    out[M::NA + 1] = __longlong_as_double((long long)(unsigned)esum);
}

// A whole tile by one warp: acc, prod and esum of the lane.
template <class M, bool W>
__device__ __forceinline__ void solo_tile(const typename M::Record& c, const MathTables* mt, const Cols& cols,
                                          int64_t tbase, int64_t ev1, typename M::Slow* sbuf, double* wbuf, int lane,
                                          double* acc, double* prod, int* esum) {
    FastScale sc;
    bool plain = !M::usable(c, ev1 - tbase, &sc);
    if (!plain) {
        const int base = sc.top;
        int run = W ? kNoWeight : 0;
        plain = !scale_to<M>(&sc, base, run);
        FastSums<M::kSums, M::kInts> s;
        clear(s);
        double tot[M::kSums], tprod = 1.0;
#pragma unroll
        for (int i = 0; i < M::kSums; ++i) tot[i] = 0.0;
#pragma unroll 1
        for (int i0 = 0; !plain && i0 < kPerLane && tbase + 32 * i0 < ev1; i0 += kSub) {
            if (W) {
                const int next = max(run, weight_exponent<true>(cols, tbase, i0, ev1, wbuf, lane));
                raise_scale(s, run, next);
                run = next;
                if (!scale_to<M>(&sc, base, run)) {
                    plain = true;
                    break;
                }
            }
            M::template quarter<W>(c, mt, cols, tbase, i0, ev1, sbuf, wbuf, lane, sc, s);
            if (W) plain = __any_sync(0xffffffffu, M::bad(c, sc, s));
#pragma unroll
            for (int i = 0; i < M::kSums; ++i) {
                tot[i] += s.f[i];
                s.f[i] = 0.0;
            }
            tprod *= s.prod;
            s.prod = 1.0;
        }
        if (!plain) {
            if (!W) plain = __any_sync(0xffffffffu, M::bad(c, sc, s));
            plain = plain || too_small<M>((int)__reduce_max_sync(0xffffffffu, (unsigned)s.most), sc, run);
        }
#pragma unroll
        for (int i = 0; i < M::kSums; ++i) s.f[i] = tot[i];
        M::accumulators(c, sc, s, acc);
        *prod = tprod;
        *esum = s.esum;
    }
    if (plain) {
        double q[M::NA + 2];                         // (apart from acc, which stays in registers)
        plain_quarters<M, W>(c, mt, cols, 0, kPerLane, tbase, ev1, sbuf, lane, q);
#pragma unroll
        for (int a = 0; a < M::NA; ++a) acc[a] = q[a];
        *prod = q[M::NA];
        *esum = (int)__double_as_longlong(q[M::NA + 1]);
    }
}

// Doubles a lane exchanges: the sums of either path, the product and the exponents.
template <class M>
constexpr int team_words() {
    return (M::kSums + M::kInts > M::NA ? M::kSums + M::kInts : M::NA) + 2;
}
template <class M, bool W>
constexpr size_t team_smem() {
    return sizeof(double) * 2 * kTeam * team_words<M>() * 32 + sizeof(typename M::Slow) * kTeam * kSub * 32 +
           sizeof(typename M::Record) + (W ? sizeof(double) * kTeam * kSub * 32 : 0);
}

// One tile per block and take, a quarter per warp.  The next take is fetched while a tile is
// in work; the exchange buffer is used in turns, so that one barrier per tile orders its
// writes after the reads of two tiles before, and the warps take turns in adding a tile up.
template <class M, bool W>
__global__ void __launch_bounds__(32 * kTeam, 4)
team_kernel(Cols cols, int64_t n, const int64_t* __restrict__ seg_begin, const int64_t* __restrict__ seg_end,
            const int64_t* __restrict__ seg_tiles, int n_seg, const Consts* __restrict__ consts,
            double* __restrict__ partials, unsigned* __restrict__ counters, unsigned* __restrict__ gcount,
            unsigned* __restrict__ work, double* __restrict__ out, int n_par) {
    constexpr int kWords = team_words<M>();
    const int out_stride = 1 + n_par;
    __shared__ MathTables mt;
    __shared__ int64_t s_take[2];
    __shared__ __align__(16) int s_most[2][kTeam];   // a quarter's largest factor, or kBad: redo the tile
    __shared__ int s_run[2];                         // the tile's largest weight
    constexpr int kBad = 0x7FFFFFFF;
    static_assert(kTeam == 4, "the quarters' largest factors are read as one word");
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    double* const xbuf = reinterpret_cast<double*>(dyn_smem);               // [2][kTeam][kWords][32]
    typename M::Slow* const sbuf =
        reinterpret_cast<typename M::Slow*>(xbuf + 2 * kTeam * kWords * 32) + wib * (kSub * 32);
    typename M::Record& c = *reinterpret_cast<typename M::Record*>(
        reinterpret_cast<typename M::Slow*>(xbuf + 2 * kTeam * kWords * 32) + kTeam * kSub * 32);

    double* const wbuf = reinterpret_cast<double*>(&c + 1) + wib * (kSub * 32);

    load_math_tables(&mt);
    // a programmatic dependent of the constants kernel: wait for its results
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
    if (threadIdx.x == 0) s_take[0] = (int64_t)atomicAdd(work, 1u);
    __syncthreads();
    int cur = -1;
    for (int turn = 0;; ++turn) {
        const int64_t tile = s_take[turn & 1];
        if (tile >= total) break;
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
        if (seg != cur) {                            // (the same for the whole block)
            __syncthreads();
            const double* src = reinterpret_cast<const double*>(consts + seg);
            double* dst = reinterpret_cast<double*>(&c);
            for (int i = threadIdx.x; i < (int)(sizeof(c) / sizeof(double)); i += blockDim.x) dst[i] = __ldg(src + i);
            __syncthreads();
            cur = seg;
        }
        const int64_t tbase = ev0 + (tile - t0) * kTile;
        double* const x = xbuf + (size_t)(turn & 1) * kTeam * kWords * 32 + lane;
        double* const own = x + wib * kWords * 32;
        const int i0 = wib * kSub;
        FastScale sc;
        bool plain = !M::usable(c, ev1 - tbase, &sc);
        const int base = sc.top;
        int run = 0;
        if (W) {
            run = kNoWeight;
            for (int j = 0; j <= i0; j += kSub) run = max(run, weight_exponent<false>(cols, tbase, j, ev1, wbuf, lane));
        }
        plain = !scale_to<M>(&sc, base, run) || plain;
        {
            FastSums<M::kSums, M::kInts> s;
            clear(s);
            if (!plain && tbase + 32 * i0 < ev1) {
                M::template quarter<W>(c, &mt, cols, tbase, i0, ev1, sbuf, wbuf, lane, sc, s);
                plain = M::bad(c, sc, s);
            }
            const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)(plain ? kBad : s.most));
            if (lane == 0) s_most[turn & 1][wib] = most;
            if (W && threadIdx.x == 32 * (kTeam - 1)) s_run[turn & 1] = run;
#pragma unroll
            for (int i = 0; i < M::kSums; ++i) own[i * 32] = s.f[i];
#pragma unroll
            for (int i = 0; i < M::kInts; ++i) own[(M::kSums + i) * 32] = __longlong_as_double(s.g[i]);
            own[(kWords - 2) * 32] = s.prod;
            own[(kWords - 1) * 32] = __longlong_as_double((long long)run << 32 | (unsigned)s.esum);
        }
        if (threadIdx.x == 32 * ((turn + 2) & (kTeam - 1))) s_take[(turn + 1) & 1] = (int64_t)atomicAdd(work, 1u);
        __syncthreads();
        {
            const int4 q = *reinterpret_cast<const int4*>(s_most[turn & 1]);
            const int most = max(max(q.x, q.y), max(q.z, q.w));
            if (W) run = s_run[turn & 1];
            FastScale t;
            scale_to<M>(&t, base, run);
            plain = most == kBad || too_small<M>(most, t, run);
        }
        if (plain) {
            double q[M::NA + 2];
            plain_quarters<M, W>(c, &mt, cols, i0, i0 + kSub, tbase, ev1, sbuf, lane, q);
#pragma unroll
            for (int a = 0; a < M::NA; ++a) own[a * 32] = q[a];
            own[(kWords - 2) * 32] = q[M::NA];
            own[(kWords - 1) * 32] = q[M::NA + 1];
            __syncthreads();
        }
        if (wib != (turn & (kTeam - 1))) continue;

        double acc[M::NA], prod = 1.0;
        int esum = 0;
        if (!plain) {
            FastSums<M::kSums, M::kInts> s;
            clear(s);
#pragma unroll
            for (int w = 0; w < kTeam; ++w) {
                const double* y = x + w * kWords * 32;
                const long long k = __double_as_longlong(y[(kWords - 1) * 32]);
                if (W) {
                    if (w) raise_scale(s, run, (int)(k >> 32));
                    run = (int)(k >> 32);
                }
                esum += (int)k;
#pragma unroll
                for (int i = 0; i < M::kSums; ++i) s.f[i] += y[i * 32];
#pragma unroll
                for (int i = 0; i < M::kInts; ++i) s.g[i] += __double_as_longlong(y[(M::kSums + i) * 32]);
                prod *= y[(kWords - 2) * 32];
            }
            scale_to<M>(&sc, base, run);
            M::accumulators(c, sc, s, acc);
        } else {
#pragma unroll
            for (int a = 0; a < M::NA; ++a) acc[a] = 0.0;
#pragma unroll 1
            for (int w = 0; w < kTeam; ++w) {
                const double* y = x + w * kWords * 32;
#pragma unroll
                for (int a = 0; a < M::NA; ++a) acc[a] += y[a * 32];
                prod *= y[(kWords - 2) * 32];
                esum += (int)__double_as_longlong(y[(kWords - 1) * 32]);
            }
        }
        acc[0] += log_of(prod, esum, &mt);
        const double share = warp_butterfly<M::NA>(acc, lane);
        if (!tile_commit<M::NA>(share, lane, tile, t0, t1, seg, partials, gcount, counters, acc)) continue;
        M::finish(c, acc, n_par, out + (size_t)seg * out_stride, lane);
        if (lane == 0) counters[seg] = 0u;
    }
    work_done(work, lane);
}

// Resident blocks per SM of a team kernel (0: not to be launched), per device.
template <class M, bool W>
int team_blocks_per_sm() {
    static int occ[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    int& per_sm = occ[dev & 63];
    if (per_sm == 0) {
        auto kern = team_kernel<M, W>;
        int v = 0;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)team_smem<M, W>()) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kern, 32 * kTeam, team_smem<M, W>()) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        per_sm = v;
    }
    return per_sm;
}

// Whether a launch over n events in n_seg segments goes to the teams: the built-in geometry (a
// tuned or given one is for single warps), and
//   * the tiles are resident at once (a team takes a quarter of a single warp's time), or
//   * at most eight per SM and two thirds full on average: a second wave of teams costs as much as
//     the first whatever its tiles hold, and short segments leave warps of a team idle.
// Measured, single warps / teams in us for 1D, 4D, tagged.  Full tiles: 300 35 / 25, 61 / 37, 81 / 47;
// 608 37 / 29, 62 / 42, 84 / 70; 1000 40 / 38, 66 / 58, 94 / 88; 1216 43 / 41, 74 / 65, 100 / 98; 1520 45 / 47,
// 76 / 75, 108 / 115.  Segments of 300 events: 608 of them 46 / 39, 66 / 52, 86 / 87; 900 51 / 57, 74 / 80,
// 95 / 97.  Of 20 events: 600 42 / 35, 61 / 50, 67 / 66; 1000 52 / 55, 73 / 83, 76 / 92.
// Segments below M::kPlainBelow events take the plain loop in either form: a warp each while there
// are at most as many as SMs (4D, 1, 30 and 100 segments of 20 events: 31 / 35, 37 / 41, 38 / 42; 200 of
// them, two to an SM, 55 / 44).
constexpr int kTeamTilesPerSm = 8;
template <class M, bool W>
bool launch_team_ok(const LaunchCfg& cfg, int64_t n, int n_seg) {
    if (cfg.warps_per_block != 1 || cfg.warps_per_sm != 0 || cfg.tiles_per_take != 1) return false;
    const int64_t sms = sm_count(), guess = tile_estimate(n, n_seg);
    const int64_t tiles = n_seg > 1 && guess < n_seg ? n_seg : guess;      // a segment has one at least
    if (n < (int64_t)n_seg * M::kPlainBelow && tiles <= sms) return false;
    const int64_t per_sm = team_blocks_per_sm<M, W>();
    return per_sm > 0 && (tiles <= per_sm * sms || (tiles <= kTeamTilesPerSm * sms && 3 * n >= 2 * kTile * tiles));
}

template <class M, bool W>
ipa_status launch_team(const Cols& cols, int64_t n, const int64_t* seg_begin, const int64_t* seg_end,
                       const int64_t* seg_tiles, int n_seg, const Consts* consts, Scratch* sc, double* out, int n_par,
                       int64_t tiles, cudaStream_t st) {
    auto kern = team_kernel<M, W>;
    constexpr size_t smem = team_smem<M, W>();
    const int per_sm = team_blocks_per_sm<M, W>();
    int64_t grid = (int64_t)per_sm * sm_count();
    if (seg_begin == nullptr && tiles < grid) grid = tiles < 1 ? 1 : tiles;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)grid);
    lc.blockDim = dim3(32 * kTeam);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    // blocks may start (and load their tables) while the constants kernel is still running
    cudaLaunchAttribute la[1];
    la[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    la[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = la;
    lc.numAttrs = 1;
    return cuda_fail(cudaLaunchKernelEx(&lc, kern, cols, n, seg_begin, seg_end, seg_tiles, n_seg, consts, sc->partials,
                                        sc->counters, sc->gcount, sc->work, out, n_par),
                     "likelihood kernel launch");
}

}  // namespace ipa
