// The accept-reject machinery of the generators (Sec. 7, Example 5), shared by
// every model: candidates tested in parallel by all SMs, kept in candidate
// order.
//
// A toy keeps its first n_sig accepted candidates in increasing candidate
// index.  Candidates are cut into chunks of kGenChunk; a block takes chunks
// from a ticket counter (toys one after another, a toy's chunks in order),
// counts what its chunk accepts, learns how many the toy's earlier chunks
// accepted by the decoupled look-back of Merrill and Garland ("Single-pass
// parallel prefix scan with decoupled look-back", 2016), and writes its events
// from there on.  How many chunks a toy needs is predicted from the model's
// acceptance (its normalisation over the envelope's) plus three standard
// deviations; in the rare toy that needs more, the block of its last chunk
// goes on alone.  The toy's events do not depend on any of this.
//
// Why: one block per toy, as before, left 151 of 152 SMs idle for a single
// sample (133 725 events of the 4D model: 30.2 ms, all of it in one block) and
// half of them in a batch of about a hundred toys.
//
// Within a chunk a warp owns 512 candidates and decides them in up to three
// passes, so that no lane waits for another's rare branch: quick() in FP32 on
// every candidate (most are rejected here), test32() in FP32 on the packed
// rest, test64() on the few that lie within the FP32 error bound of their
// threshold.  A decision is always the FP64 test's: quick() and test32()
// decide only outside the bound.  Before, the angular test of the tenth of
// the candidates that pass the time test ran in almost every iteration of a
// warp with three lanes active.  (Packed or not, the FP64 tests cost a warp the
// same: hence the last pass.)
#pragma once

#include <stdint.h>

#include "int_math.cuh"
#include "ipa_internal.cuh"
#include "philox.cuh"
#include "tile_reduce.cuh"

namespace ipa {

constexpr int kGenWarps = kBlock / 32;
constexpr int kGenPerLane = 16;                            // candidates per lane and chunk
constexpr int kGenWarpCand = 32 * kGenPerLane;             // 512
constexpr int kGenChunk = kGenWarps * kGenWarpCand;        // 4096
constexpr int kGenWords = kGenChunk / 32;                  // words of the chunk's bit mask
constexpr int kBkgChunk = 2048;                            // background events per ticket
// A toy is cut into chunks only where a chunk accepts at least this many events
// on average: the look-back's status words then stay below one byte per event.
constexpr int kGenMinKept = 16;

// What a test says of a candidate.
enum GenCode { kDrop = 0, kKeep = 1, kTest32 = 2, kTest64 = 3 };

struct GenArgs {
    ModelDev m;
    const Consts* consts;
    uint32_t k0, k1;
    int n_toys;
    const int64_t *n_sig, *n_bkg, *offsets;
    int64_t capacity;
    double *t, *ck, *cl, *phi, *q;
    // ticket prefix per toy (n_toys + 1), the ticket counter and one status word
    // per ticket; base == nullptr: no workspace, one block per toy
    const int64_t* base;
    unsigned long long* ticket;
    unsigned long long* status;
};

// (v + 1) 2^-53 and 2 (v + 1) 2^-53 - 1 for the 53-bit v of two words, exactly,
// by integer operations (u01 and 2 u01 - 1 cost two and four FP64 instructions).
__device__ __forceinline__ unsigned long long u53(uint32_t a, uint32_t b) {
    return (((((unsigned long long)a) << 32) | b) >> 11) + 1ull;
}
__device__ __forceinline__ double u01_int(uint32_t a, uint32_t b) {
    return q62_to_double_nb((long long)(u53(a, b) << 9), 0);
}
__device__ __forceinline__ double sym_int(uint32_t a, uint32_t b) {
    return q62_to_double_nb((long long)(u53(a, b) << 10) - kOneQ62, 0);
}

constexpr float kTwoM32 = 2.3283064365386963e-10f;   // 2^-32
constexpr float kUlp2 = 4.76837158203125e-07f;       // 2^-21
constexpr float kUlp1 = 2.384185791015625e-07f;      // 2^-22: one FP32 rounding with a factor 2 to spare

// u ~ a 2^-32 from the high word of a uniform: |u32 - u| <= 2^-24 u + 2^-31.
__device__ __forceinline__ float u32of(uint32_t hi) { return __uint2float_rn(hi) * kTwoM32; }

// A decision from u M against a value v known to +-err: +-(u M's own error) included.
__device__ __forceinline__ GenCode decide32(float lhs, float dl, float v, float err) {
    if (lhs + dl < v - err) return kKeep;
    if (lhs - dl > v + err) return kDrop;
    return kTest64;                                  // also NaN
}

struct GenLists {
    uint16_t l32[kGenWarps][kGenWarpCand];
    uint16_t l64[kGenWarps][kGenWarpCand];
    uint32_t keep[kGenWords];
    int before[kGenWords + 1];     // accepted before each word of keep
    int64_t take;
    int64_t got;
};

// Decide the chunk's candidates j0 .. j0 + kGenChunk: bit mask and its prefix
// in L; returns the number accepted.  Block-collective.
template <class G>
__device__ __noinline__ int gen_count(const typename G::Shared& S, GenLists& L, uint64_t j0, uint32_t toy, uint32_t k0, uint32_t k1) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const uint64_t jw = j0 + (uint64_t)w * kGenWarpCand;
    int n32 = 0, n64 = 0;
    if (lane < kGenPerLane) L.keep[w * kGenPerLane + lane] = 0u;
    __syncwarp();
#pragma unroll 1
    for (int i = 0; i < kGenPerLane; ++i) {
        const int cand = i * 32 + lane;
        const GenCode c = G::quick(S, jw + cand, toy, k0, k1);
        if (G::kQuickKeeps) {
            const unsigned k = __ballot_sync(0xffffffffu, c == kKeep);
            if (lane == 0) L.keep[w * kGenPerLane + i] = k;
        }
        const unsigned a = __ballot_sync(0xffffffffu, c == kTest32);
        if (c == kTest32) L.l32[w][n32 + __popc(a & below)] = (uint16_t)cand;
        n32 += __popc(a);
        const unsigned b = __ballot_sync(0xffffffffu, c == kTest64);
        if (c == kTest64) L.l64[w][n64 + __popc(b & below)] = (uint16_t)cand;
        n64 += __popc(b);
    }
    __syncwarp();
    for (int x0 = 0; x0 < n32; x0 += 32) {
        const int x = x0 + lane;
        const int cand = x < n32 ? L.l32[w][x] : 0;
        const GenCode c = x < n32 ? G::test32(S, jw + cand, toy, k0, k1) : kDrop;
        if (c == kKeep) atomicOr(&L.keep[w * kGenPerLane + (cand >> 5)], 1u << (cand & 31));
        const unsigned b = __ballot_sync(0xffffffffu, c == kTest64);
        if (c == kTest64) L.l64[w][n64 + __popc(b & below)] = (uint16_t)cand;
        n64 += __popc(b);
    }
    __syncwarp();
    for (int x = lane; x < n64; x += 32) {
        const int cand = L.l64[w][x];
        if (G::test64(S, jw + cand, toy, k0, k1)) atomicOr(&L.keep[w * kGenPerLane + (cand >> 5)], 1u << (cand & 31));
    }
    __syncthreads();
    if (w == 0) {
        constexpr int kPer = kGenWords / 32;
        int c[kPer], s = 0;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            c[i] = s;
            s += __popc(L.keep[lane * kPer + i]);
        }
        int x = s;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, d);
            if (lane >= d) x += y;
        }
#pragma unroll
        for (int i = 0; i < kPer; ++i) L.before[lane * kPer + i] = x - s + c[i];
        if (lane == 31) L.before[kGenWords] = x;
    }
    __syncthreads();
    return L.before[kGenWords];
}

// Write the chunk's accepted candidates as events got, got + 1, ... of the toy.
template <class G>
__device__ __noinline__ void gen_write(const typename G::Shared& S, const GenArgs& A, const GenLists& L, uint64_t j0, uint32_t toy,
                          int64_t got, int64_t ns, int64_t off) {
    const int total = L.before[kGenWords];
    for (int k = threadIdx.x; k < total; k += kBlock) {
        if (got + k >= ns) break;
        int lo = 0, hi = kGenWords - 1;
        while (lo < hi) {                            // the last word with before <= k
            const int mid = (lo + hi + 1) >> 1;
            if (L.before[mid] <= k) lo = mid; else hi = mid - 1;
        }
        const int bit = nth_set(L.keep[lo], k - L.before[lo]);
        G::signal(S, A, j0 + lo * 32 + bit, toy, off + got + k);
    }
}

// Status word of a ticket: the count its chunk accepted (kAggregate) or the
// toy's count up to and with it (kPrefix), in the bits above the two flag bits.
enum : unsigned long long { kAggregate = 1ull, kPrefix = 2ull };
constexpr int kLookBackPolls = 1 << 20;

// Events the toy accepted before chunk `local` (ticket tk), having published
// this chunk's count.  Called by warp 0.  The blocks of the earlier tickets are
// running (tickets are handed out in order), so every word waited for gets
// written; the wait is bounded all the same: returns -1 when it runs out.
__device__ __forceinline__ int64_t look_back(unsigned long long* status, int64_t tk, int64_t local, int count, int lane) {
    volatile unsigned long long* st = status;
    if (lane == 0) st[tk] = ((unsigned long long)count << 2) | (local == 0 ? kPrefix : kAggregate);
    if (local == 0) return 0;
    int64_t sum = 0;
    int64_t at = tk - 1;                             // the window is at, at - 1, ..., at - 31
    const int64_t first = tk - local;
    int polls = 0;
    while (true) {
        const int64_t mine = at - lane;
        unsigned long long v = kPrefix;
        if (mine >= first) v = st[mine];
        while (__any_sync(0xffffffffu, (v & 3ull) == 0ull)) {
            if (++polls > kLookBackPolls) return -1;
            __nanosleep(40);
            if ((v & 3ull) == 0ull) v = st[mine];
        }
        const unsigned full = __ballot_sync(0xffffffffu, (v & 3ull) == kPrefix);
        const int stop = full ? __ffs(full) - 1 : 31;
        int64_t x = lane <= stop ? (int64_t)(v >> 2) : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        sum += x;
        if (full) break;
        at -= 32;
    }
    if (lane == 0) st[tk] = ((unsigned long long)(sum + count) << 2) | kPrefix;
    return sum;
}

// The signal of one toy from candidate j0 on, `got` events already kept: chunk
// after chunk by this block, then NaN for what the candidate budget left open.
template <class G>
__device__ void gen_rest(const typename G::Shared& S, const GenArgs& A, GenLists& L, uint64_t j0, uint32_t toy,
                         int64_t got, int64_t ns, int64_t off, bool usable) {
    // non-finite or non-positive envelopes (non-physical theta) accept nothing:
    // the signal is then filled with NaN instead of searched for forever
    const uint64_t budget = usable ? (uint64_t)ns * 65536ull + (1ull << 22) : 0ull;
    for (; got < ns && j0 < budget; j0 += kGenChunk) {
        __syncthreads();
        const int n = gen_count<G>(S, L, j0, toy, A.k0, A.k1);
        gen_write<G>(S, A, L, j0, toy, got, ns, off);
        got += n;
    }
    for (int64_t pos = got + threadIdx.x; pos < ns; pos += kBlock) G::fill_nan(A, off + pos);
}

__device__ __forceinline__ bool gen_toy(const GenArgs& A, int toy, int64_t* ns, int64_t* nb, int64_t* off) {
    *ns = A.n_sig[toy];
    *nb = A.n_bkg[toy];
    *off = A.offsets[toy];
    return !(*ns < 0 || *nb < 0 || *off < 0 || *off + *ns + *nb > A.capacity);   // else skipped
}

template <class G>
__global__ void __launch_bounds__(kBlock, G::kBlocksPerSm) generate_kernel(GenArgs A) {
    __shared__ typename G::Shared S;
    __shared__ GenLists L;
    G::setup(S, A);
    __syncthreads();
    const bool usable = G::usable(S);
    if (A.base == nullptr) {
        for (int toy = blockIdx.x; toy < A.n_toys; toy += gridDim.x) {
            int64_t ns, nb, off;
            if (!gen_toy(A, toy, &ns, &nb, &off)) continue;
            gen_rest<G>(S, A, L, 0, (uint32_t)toy, 0, ns, off, usable);
            for (int64_t i = threadIdx.x; i < nb; i += kBlock) G::background(S, A, (uint64_t)i, (uint32_t)toy, off + ns + i);
        }
        return;
    }
    const int64_t total = A.base[A.n_toys];
    while (true) {
        __syncthreads();                             // L is free
        if (threadIdx.x == 0) L.take = (int64_t)atomicAdd(A.ticket, 1ull);
        __syncthreads();
        const int64_t tk = L.take;
        if (tk >= total) break;
        const int toy = find_segment(A.base, A.n_toys, tk);
        const int64_t t0 = A.base[toy], n_chunks = A.base[toy + 1] - t0;
        int64_t ns, nb, off;
        gen_toy(A, toy, &ns, &nb, &off);
        const int64_t n_sig_chunks = n_chunks - (nb + kBkgChunk - 1) / kBkgChunk;
        const int64_t local = tk - t0;
        if (local >= n_sig_chunks) {
            const int64_t i0 = (local - n_sig_chunks) * kBkgChunk;
            const int64_t i1 = i0 + kBkgChunk < nb ? i0 + kBkgChunk : nb;
            for (int64_t i = i0 + threadIdx.x; i < i1; i += kBlock)
                G::background(S, A, (uint64_t)i, (uint32_t)toy, off + ns + i);
            continue;
        }
        const uint64_t j0 = (uint64_t)local * kGenChunk;
        int n = usable ? gen_count<G>(S, L, j0, (uint32_t)toy, A.k0, A.k1) : 0;
        int64_t got = 0;
        if (n_sig_chunks > 1) {                      // (tickets beyond the status words are toys of one chunk)
            if (threadIdx.x < 32) {
                const int64_t before = look_back(A.status, tk, local, n, threadIdx.x);
                if (threadIdx.x == 0) L.got = before;
            }
            __syncthreads();
            got = L.got;
        }
        if (got < 0) {                               // the wait ran out: count the earlier chunks here
            got = 0;
            for (int64_t c = 0; c < local; ++c) {
                got += gen_count<G>(S, L, (uint64_t)c * kGenChunk, (uint32_t)toy, A.k0, A.k1);
                __syncthreads();
            }
            n = gen_count<G>(S, L, j0, (uint32_t)toy, A.k0, A.k1);
        }
        if (n > 0) gen_write<G>(S, A, L, j0, (uint32_t)toy, got, ns, off);
        if (local == n_sig_chunks - 1)
            gen_rest<G>(S, A, L, j0 + kGenChunk, (uint32_t)toy, got + n, ns, off, usable);
    }
}

// Tickets per toy and their prefix (one block).  Signal chunks: enough for
// n_sig + 3 sqrt(n_sig) + 8 accepted candidates at the model's acceptance;
// one (whose block goes on alone) where a chunk accepts fewer than
// kGenMinKept, or where the total would exceed max_tickets.
template <class G>
__global__ void gen_tickets_kernel(GenArgs A, int64_t max_tickets, int64_t* __restrict__ base) {
    __shared__ int64_t run[1024];
    __shared__ float per_chunk;
    G::acceptance(A, &per_chunk);
    __syncthreads();
    const float kept = per_chunk * (float)kGenChunk;
    const int nt = blockDim.x;
    const int per = (A.n_toys + nt - 1) / nt;
    const int b = min(A.n_toys, (int)threadIdx.x * per), e = min(A.n_toys, b + per);
    for (int round = 0; round < 2; ++round) {
        const bool split = round == 0 && kept >= (float)kGenMinKept && kept <= 2.0f * kGenChunk;
        auto tickets = [&](int toy) -> int64_t {
            int64_t ns, nb, off;
            if (!gen_toy(A, toy, &ns, &nb, &off)) return 0;
            int64_t c = ns > 0;
            if (split && ns > 0) {
                const float f = (float)ns;
                c = (int64_t)ceilf((f + 3.0f * sqrtf(f) + 8.0f) / kept);
                if (c < 1) c = 1;
            }
            return c + (nb + kBkgChunk - 1) / kBkgChunk;
        };
        int64_t sum = 0;
        for (int s = b; s < e; ++s) sum += tickets(s);
        __syncthreads();
        run[threadIdx.x] = sum;
        __syncthreads();
        for (int d = 1; d < nt; d <<= 1) {
            const int64_t v = (int)threadIdx.x >= d ? run[threadIdx.x - d] : 0;
            __syncthreads();
            run[threadIdx.x] += v;
            __syncthreads();
        }
        if (round == 0 && run[nt - 1] > max_tickets) continue;
        int64_t acc = threadIdx.x ? run[threadIdx.x - 1] : 0;
        for (int s = b; s < e; ++s) {
            base[s] = acc;
            acc += tickets(s);
        }
        if ((int)threadIdx.x == nt - 1) base[A.n_toys] = run[nt - 1];
        break;
    }
}

// consts.cu's record is in place on the stream.  The workspace (ticket prefix,
// counter, status words) is allocated in stream order and given back after the
// kernel; without it (no memory) a block generates a toy alone, with the same
// events.
template <class G>
ipa_status launch_generator(GenArgs A, cudaStream_t s) {
    int dev = 0;
    cudaGetDevice(&dev);
    static int occ[64] = {};
    int& per_sm = occ[dev & 63];
    if (per_sm == 0) {
        int v = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, generate_kernel<G>, kBlock, 0);
        per_sm = e == cudaSuccess && v >= 1 ? v : 1;
    }
    // (n_sig + 3 sqrt(n_sig) + 8) / kGenMinKept + 2 <= n_sig / 10 + 3, and one per kBkgChunk background events
    const int64_t max_tickets = A.capacity / 10 + 4 * (int64_t)A.n_toys + A.capacity / kBkgChunk + 1;
    const size_t words = (size_t)A.n_toys + 2 + (size_t)max_tickets;
    void* ws = nullptr;
    const int64_t most = (int64_t)sm_count() * per_sm;
    if (pool_alloc(&ws, words * 8, s, "generator workspace") == IPA_OK) {
        ipa_status st = cuda_fail(cudaMemsetAsync(ws, 0, words * 8, s), "generator workspace reset");
        int64_t* base = static_cast<int64_t*>(ws);
        A.base = base;
        A.ticket = reinterpret_cast<unsigned long long*>(base + A.n_toys + 1);
        A.status = A.ticket + 1;
        if (st == IPA_OK) {
            gen_tickets_kernel<G><<<1, 1024, 0, s>>>(A, max_tickets, base);
            generate_kernel<G><<<(unsigned)(max_tickets < most ? max_tickets : most), kBlock, 0, s>>>(A);
            st = cuda_fail(cudaGetLastError(), "toygen kernel launch");
        }
        pool_free(ws, s);
        return st;
    }
    cudaGetLastError();
    A.base = nullptr;
    generate_kernel<G><<<(unsigned)A.n_toys, kBlock, 0, s>>>(A);
    return cuda_fail(cudaGetLastError(), "toygen kernel launch");
}

}  // namespace ipa
