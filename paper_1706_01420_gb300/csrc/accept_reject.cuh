// The accept-reject machinery of the generators (Sec. 7, Example 5), shared by
// every model: candidates tested in parallel by all SMs, kept in candidate
// order.
//
// A toy keeps its first n_sig accepted candidates in increasing candidate
// index.  Candidates are cut into chunks; a warp takes chunks from a ticket
// counter (toys one after another, a toy's chunks in order), counts what its
// chunk accepts, learns how many the toy's earlier chunks accepted by the
// decoupled look-back of Merrill and Garland ("Single-pass parallel prefix scan
// with decoupled look-back", 2016), and writes its events from there on.  How
// many chunks a toy needs is predicted from the model's acceptance (its
// normalisation over the envelope's) plus three standard deviations; in the
// rare toy that needs more, the warp of its last chunk goes on alone.  The
// toy's events do not depend on any of this.
//
// Why: one block per toy, as before, left 151 of 152 SMs idle for a single
// sample (133 725 events of the 4D model: 30.2 ms, all of it in one block) and
// half of them in a batch of about a hundred toys.  A warp per chunk, not a
// block: with 4096 candidates per block the warps spent half of their time at
// the block's barriers (waiting for the look-back, for the one warp with an
// FP64 test and for each other).
//
// A warp decides 1024 candidates in up to three passes, so that no lane waits
// for another's rare branch: quick() in FP32 on every candidate (most are
// rejected here), test32() in FP32 on the packed rest, test64() on the few that
// lie within the FP32 error bound of their threshold.  A decision is always
// the FP64 test's: quick() and test32() decide only outside the bound.
// Before, the angular test of the tenth of the candidates that pass the time
// test ran in almost every iteration of a warp with three lanes active.
//
// Bound: instruction issue (about 155 warp instructions per 32 candidates, 45 of
// them Philox's and the first test's, 18 of those 32 x 32 -> 64-bit products; a 4D
// event needs 50 candidates) and, where tickets are small, the latency of the
// look-back: 67 % of the issue slots busy.  Measured (one block per toy / blocks with
// barriers / warps / the first test folded into one multiply-add and compare on the
// words, two candidates at once, and larger tickets where there are many): 4D,
// one sample of 133 725 events 30.2 ms / 92 us / 84 us / 81 us; 4D, 512 toys of
// Poisson(2e4) 11.5 / 4.5 / 3.7 / 2.8 ms; phi_s, 102 toys of 8170 (every candidate in
// FP64 before) 24.0 / 0.77 / 0.68 / 0.69 ms.
#pragma once

#include <stdint.h>

#include "int_math.cuh"
#include "ipa_internal.cuh"
#include "philox.cuh"
#include "tile_reduce.cuh"

namespace ipa {

constexpr int kGenWarps = kBlock / 32;
constexpr int kGenCand = 1024;           // candidates a warp decides at once: 32 words of its bit mask
constexpr int kGenPick = 256;            // accepted candidates listed at once for writing
constexpr int kBkgChunk = 512;           // background events per ticket
// A ticket is 1, 2, 4, ... kGenMaxSub times kGenCand candidates, as many as
// accept kGenMinKept events on average: the look-back's status words then
// stay below 1.3 bytes per event.  A toy of an envelope that accepts less is
// one ticket: a warp alone (with tickets of at most 64 units, a range of 2e4
// lifetimes was one: 300 1D events 624 ms, 142 at a block per toy).
constexpr int kGenMinKept = 8;
// ... and more where there is work enough: while kGenPerWarp tickets per resident
// warp are left and a ticket's events fit the list (kGenPick) with room to spare.
// Fewer look-backs: the 512 toys take 3.19 ms at one unit per ticket, 2.88 at two and
// 2.76 at four; a single sample of 133 725 events, with 1.4 units per warp, 82, 91
// and 102 us.
constexpr int kGenMostKept = 160;
constexpr int kGenPerWarp = 16;
constexpr int kGenMaxSub = 1 << 12;      // a tenth of a second of one warp; acceptances down to 2e-6 are cut

// What a test says of a candidate.
enum GenCode { kDrop = 0, kKeep = 1, kTest32 = 2, kTest64 = 3 };

struct GenArgs {
    ModelDev m;
    const Consts* consts;
    PhiloxKeys keys;
    int n_toys;
    const int64_t *n_sig, *n_bkg, *offsets;
    int64_t capacity;
    double *t, *ck, *cl, *phi, *q;
    // ticket prefix per toy (n_toys + 1 entries, then kGenCand units per ticket),
    // the ticket counter and one status word per ticket; base == nullptr: no
    // workspace, one warp per toy
    const int64_t* base;
    unsigned long long* ticket;
    unsigned long long* status;
};

// Candidate or background event `lo` + 2^32 hi of a toy.
struct GenIdx {
    uint32_t lo, hi, toy;
};

__device__ __forceinline__ U4 gen_draw(const GenArgs& A, const GenIdx& j, uint32_t call) {
    return keyed(A.keys, j.lo, j.hi, j.toy, call);
}

// (v + 1) 2^-53 and 2 (v + 1) 2^-53 - 1 for the 53-bit v of two words, exactly,
// by integer operations (a conversion, a product and a sum would be two and four FP64 instructions).
__device__ __forceinline__ unsigned long long u53(uint32_t a, uint32_t b) {
    return (((((unsigned long long)a) << 32) | b) >> 11) + 1ull;
}
__device__ __forceinline__ double u01_int(uint32_t a, uint32_t b) {
    return q62_to_double_nb((long long)(u53(a, b) << 9), 0);
}
__device__ __forceinline__ double sym_int(uint32_t a, uint32_t b) {
    return q62_to_double_nb((long long)(u53(a, b) << 10) - (1ll << 62), 0);
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

// One warp's lists, and its ticket's state: kept in shared memory (uniform over
// the warp), since in registers it spilled the candidates' loop.
struct GenLists {
    uint16_t l32[kGenCand];
    uint16_t l64[kGenCand];
    uint32_t pick[kGenPick];
    uint32_t keep[32];
    int64_t ns, off, got;          // the toy's signal, its first event, events accepted before unit u
    int64_t tk, local, n_chunks;   // ticket, its chunk of the toy, the toy's chunks
    int64_t c, u;                  // chunk and unit (of kGenCand candidates) in work
    int nu;                        // units decided at once
    uint32_t toy;
    bool look;                     // the look-back is to come
};

// Decide candidates j0 .. j0 + kGenCand: lane l returns the bits of candidates
// 32 l .. 32 l + 31.  Warp-collective.
template <class G>
__device__ __forceinline__ uint32_t gen_decide(const typename G::Shared& S, const GenArgs& A, GenLists& L, uint64_t j0,
                                               uint32_t toy, int lane) {
    const unsigned below = (1u << lane) - 1u;
    const uint32_t lo = (uint32_t)j0, hi = (uint32_t)(j0 >> 32);   // no carry: j0 is a multiple of kGenCand
    int n32 = 0, n64 = 0;
    uint32_t word = 0u;
    __syncwarp();
    L.keep[lane] = 0u;
#pragma unroll (G::kUnroll)
    for (int i = 0; i < 32; ++i) {
        const int cand = i * 32 + lane;
        const GenCode c = G::quick(S, A, GenIdx{lo + cand, hi, toy});
        if (G::kQuickKeeps) {
            const unsigned k = __ballot_sync(0xffffffffu, c == kKeep);
            if (lane == i) word = k;
        }
        const unsigned a = __ballot_sync(0xffffffffu, c == kTest32);
        if (c == kTest32) L.l32[n32 + __popc(a & below)] = (uint16_t)cand;
        n32 += __popc(a);
        if (G::kQuick64) {
            const unsigned b = __ballot_sync(0xffffffffu, c == kTest64);
            if (c == kTest64) L.l64[n64 + __popc(b & below)] = (uint16_t)cand;
            n64 += __popc(b);
        }
    }
    __syncwarp();
#pragma unroll 1
    for (int x0 = 0; x0 < n32; x0 += 32) {
        const int x = x0 + lane;
        GenCode c = kDrop;
        int cand = 0;
        if (x < n32) {
            cand = L.l32[x];
            c = G::test32(S, A, GenIdx{lo + cand, hi, toy});
        }
        if (c == kKeep) atomicOr(&L.keep[cand >> 5], 1u << (cand & 31));
        const unsigned b = __ballot_sync(0xffffffffu, c == kTest64);
        if (c == kTest64) L.l64[n64 + __popc(b & below)] = (uint16_t)cand;
        n64 += __popc(b);
    }
    __syncwarp();
#pragma unroll 1
    for (int x = lane; x < n64; x += 32) {
        const int cand = L.l64[x];
        if (G::test64(S, A, GenIdx{lo + cand, hi, toy})) atomicOr(&L.keep[cand >> 5], 1u << (cand & 31));
    }
    __syncwarp();
    return word | L.keep[lane];
}

// Exclusive prefix of the lanes' popcounts; *total: their sum.
__device__ __forceinline__ int gen_prefix(uint32_t word, int lane, int* total) {
    const int n = __popc(word);
    int x = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    *total = __shfl_sync(0xffffffffu, x, 31);
    return x - n;
}

// Append the candidates of `word` (first rank `pre`) whose ranks lie in [r0, r0 +
// kGenPick) to the list, as offsets from `off`.
__device__ __forceinline__ void gen_pick(GenLists& L, uint32_t word, int pre, int r0, int off, int lane) {
    for (int r = pre - r0; word && r < kGenPick; ++r) {
        const int bit = __ffs((int)word) - 1;
        word &= word - 1u;
        if (r >= 0) L.pick[r] = (uint32_t)(off + lane * 32 + bit);
    }
}

// Write listed candidates (n of them, offsets from j0) as events got, got + 1, ... of the toy.
template <class G>
__device__ __forceinline__ void gen_write(const typename G::Shared& S, const GenArgs& A, const GenLists& L, uint64_t j0,
                                          uint32_t toy, int n, int64_t got, int64_t ns, int64_t off, int lane) {
#pragma unroll 1
    for (int k = lane; k < n; k += 32) {
        if (got + k >= ns) break;
        const uint64_t j = j0 + L.pick[k];
        G::signal(S, A, GenIdx{(uint32_t)j, (uint32_t)(j >> 32), toy}, off + got + k);
    }
}

// Status word of a ticket: the count its chunk accepted (kAggregate) or the
// toy's count up to and with it (kPrefix), in the bits above the two flag bits.
enum : unsigned long long { kAggregate = 1ull, kPrefix = 2ull };
constexpr int kLookBackPolls = 1 << 20;

// Events the toy accepted before chunk `local` (ticket tk), having published
// this chunk's count.  Warp-collective.  The warps of the earlier tickets are
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

__device__ __forceinline__ bool gen_toy(const GenArgs& A, int toy, int64_t* ns, int64_t* nb, int64_t* off) {
    *ns = A.n_sig[toy];
    *nb = A.n_bkg[toy];
    *off = A.offsets[toy];
    return !(*ns < 0 || *nb < 0 || *off < 0 || *off + *ns + *nb > A.capacity);   // else skipped
}

template <class G>
__global__ void __launch_bounds__(kBlock, G::kBlocksPerSm) generate_kernel(const __grid_constant__ GenArgs A) {
    __shared__ typename G::Shared S;
    extern __shared__ __align__(16) unsigned char dyn_smem[];
    G::setup(S, A);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    GenLists& L = reinterpret_cast<GenLists*>(dyn_smem)[threadIdx.x >> 5];
    const bool usable = G::usable(S);
    const bool alone = A.base == nullptr;            // ticket k is the whole of toy k
    const int sub = alone ? 1 : (int)A.base[A.n_toys + 1];
    if (lane == 0) L.tk = (int64_t)(blockIdx.x * kGenWarps + (threadIdx.x >> 5)) - (int64_t)gridDim.x * kGenWarps;
    while (true) {
        __syncwarp();
        if (lane == 0) L.tk = alone ? L.tk + (int64_t)gridDim.x * kGenWarps : (int64_t)atomicAdd(A.ticket, 1ull);
        __syncwarp();
        const int64_t tk = L.tk;
        if (tk >= (alone ? A.n_toys : A.base[A.n_toys])) break;
        const int toy = alone ? (int)tk : find_segment(A.base, A.n_toys, tk);
        {
            int64_t ns, nb, off;
            if (!gen_toy(A, toy, &ns, &nb, &off)) continue;
            // the ticket's part of the toy: one of its signal chunks, or background events
            int64_t local = 0, n_chunks = ns > 0, i0 = 0, i1 = nb;
            if (!alone) {
                const int64_t t0 = A.base[toy];
                local = tk - t0;
                n_chunks = A.base[toy + 1] - t0 - (nb + kBkgChunk - 1) / kBkgChunk;
                i0 = local < n_chunks ? nb : (local - n_chunks) * kBkgChunk;
                i1 = i0 + kBkgChunk < nb ? i0 + kBkgChunk : nb;
            }
#pragma unroll 1
            for (int64_t i = i0 + lane; i < i1; i += 32)
                G::background(S, A, GenIdx{(uint32_t)i, (uint32_t)((uint64_t)i >> 32), (uint32_t)toy}, off + ns + i);
            if (local >= n_chunks) continue;
            if (lane == 0) {
                L.ns = ns;
                L.off = off;
                L.got = 0;
                L.local = local;
                L.n_chunks = n_chunks;
                L.c = local;
                L.u = local * sub;
                L.nu = sub;
                L.toy = (uint32_t)toy;
                L.look = n_chunks > 1;
            }
            __syncwarp();
        }
        // this ticket's chunk, and after a toy's last chunk whatever the toy still lacks
        while (true) {
            uint32_t word = 0u;
            int n = 0, pre = 0, last = 0;
            const int nu = L.nu;
            for (int s = 0; s < nu && usable; ++s) {
                word = gen_decide<G>(S, A, L, (uint64_t)(L.u + s) * kGenCand, L.toy, lane);
                pre = gen_prefix(word, lane, &last);
                if (nu > 1 && n + last <= kGenPick) gen_pick(L, word, pre + n, 0, s * kGenCand, lane);
                n += last;
            }
            __syncwarp();
            if (L.look) {
                const int64_t before = look_back(A.status, L.tk, L.local, n, lane);
                __syncwarp();
                if (lane == 0) {
                    L.look = false;
                    L.got = before < 0 ? 0 : before;
                    if (before < 0) L.c = L.u = 0;   // the wait ran out: count the toy's chunks from its first
                }
                __syncwarp();
                if (before < 0) continue;
            }
            if (L.c >= L.local) {
                if (nu > 1 && n > kGenPick) {        // more than the list holds: unit by unit
                    __syncwarp();
                    if (lane == 0) L.nu = 1;
                    __syncwarp();
                    continue;
                }
                for (int r0 = 0; r0 < n; r0 += kGenPick) {
                    __syncwarp();
                    if (nu == 1) gen_pick(L, word, pre, r0, 0, lane);
                    __syncwarp();
                    gen_write<G>(S, A, L, (uint64_t)L.u * kGenCand, L.toy, min(n - r0, kGenPick), L.got + r0, L.ns, L.off,
                                 lane);
                }
            }
            const int64_t got = L.got + n, u = L.u + nu;
            int64_t c = L.c;
            const bool ends = u >= (c + 1) * sub;    // of the chunk
            if (ends && c == L.local && L.local != L.n_chunks - 1) break;
            c += ends;
            __syncwarp();
            if (lane == 0) {
                L.got = got;
                L.u = u;
                L.c = c;
                if (ends) L.nu = sub;
            }
            __syncwarp();
            // non-finite or non-positive envelopes (non-physical theta) accept nothing:
            // the signal is then filled with NaN instead of searched for forever
            const uint64_t budget = usable ? (uint64_t)L.ns * 65536ull + (1ull << 22) : 0ull;
            if (ends && c > L.local && !(got < L.ns && (uint64_t)u * kGenCand < budget)) break;
        }
        if (L.local == L.n_chunks - 1)
            for (int64_t pos = L.got + lane; pos < L.ns; pos += 32) G::fill_nan(A, L.off + pos);
    }
}

// A block per toy, its warps 128 candidates each at a time: for the few events of G::kBlockEvents
// and fewer per toy, where a warp's 1024 candidates at once are most of the toy's and the
// tickets cost two launches.  1D, one toy of 100 / 500 / 1000 events: 37 us by tickets, 26 / 63 / 110
// by one warp, 20 / 32 / 47 so (the line is where the tickets win; an envelope that accepts little
// is walked by a block whatever it costs, as the host does not know).  2000 toys of 10 / 100: 93 / 100 us
// by tickets, 41 / 52 so; more toys than warps take a warp each (5000 of 300 and 20 000 of 500:
// 197 / 866 by tickets, 200 / 1130 by blocks, 138 / 657).
template <class G>
__global__ void __launch_bounds__(kBlock) generate_block_kernel(const __grid_constant__ GenArgs A) {
    constexpr int kRows = 4;
    __shared__ typename G::Shared S;
    __shared__ int s_kept[2][kGenWarps];
    G::setup(S, A);
    __syncthreads();
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const bool usable = G::usable(S);
    int turn = 0;
    for (int toy = blockIdx.x; toy < A.n_toys; toy += gridDim.x) {
        int64_t ns, nb, off;
        if (!gen_toy(A, toy, &ns, &nb, &off)) continue;
        for (int64_t i = threadIdx.x; i < nb; i += kBlock)
            G::background(S, A, GenIdx{(uint32_t)i, (uint32_t)((uint64_t)i >> 32), (uint32_t)toy}, off + ns + i);
        const uint64_t budget = usable ? (uint64_t)ns * 65536ull + (1ull << 22) : 0ull;    // as generate_kernel
        int64_t got = 0;
        for (uint64_t j0 = 0; got < ns && j0 < budget; j0 += kRows * kBlock, turn ^= 1) {
            const uint64_t j1 = j0 + (uint64_t)(wib * kRows * 32 + lane);
            unsigned kept[kRows];
            int n = 0;
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
                const uint64_t jr = j1 + 32u * r;
                const GenIdx j = {(uint32_t)jr, (uint32_t)(jr >> 32), (uint32_t)toy};
                GenCode c = G::quick(S, A, j);
                if (c == kTest32) c = G::test32(S, A, j);
                if (c == kTest64) c = G::test64(S, A, j) ? kKeep : kDrop;
                kept[r] = __ballot_sync(0xffffffffu, c == kKeep);
                n += __popc(kept[r]);
            }
            if (lane == 0) s_kept[turn][wib] = n;
            __syncthreads();                         // (the next round writes the other half)
            int64_t pos = got;
#pragma unroll
            for (int w = 0; w < kGenWarps; ++w) {
                const int v = s_kept[turn][w];
                pos += w < wib ? v : 0;
                got += v;
            }
#pragma unroll
            for (int r = 0; r < kRows; ++r) {
                const int64_t at = pos + __popc(kept[r] & below);
                const uint64_t jr = j1 + 32u * r;
                if ((kept[r] >> lane & 1u) && at < ns)
                    G::signal(S, A, GenIdx{(uint32_t)jr, (uint32_t)(jr >> 32), (uint32_t)toy}, off + at);
                pos += __popc(kept[r]);
            }
        }
        for (int64_t pos = got + threadIdx.x; pos < ns; pos += kBlock) G::fill_nan(A, off + pos);
    }
}

// Tickets per toy, their prefix and the candidates per ticket (one block).
// Signal chunks: enough for n_sig + 3 sqrt(n_sig) + 8 accepted candidates at the
// model's acceptance; one (whose warp goes on alone) where even the largest
// chunk accepts fewer than kGenMinKept, or where the total would exceed
// max_tickets.
template <class G>
__global__ void gen_tickets_kernel(const __grid_constant__ GenArgs A, int64_t max_tickets, int64_t n_warps,
                                   int64_t* __restrict__ base) {
    __shared__ int64_t run[1024];
    __shared__ float per_cand;
    __shared__ unsigned long long events;            // of signal, in all toys
    if (threadIdx.x == 0) events = 0ull;
    __syncthreads();
    const int nt = blockDim.x;
    const int per = (A.n_toys + nt - 1) / nt;
    const int b = min(A.n_toys, (int)threadIdx.x * per), e = min(A.n_toys, b + per);
    {
        unsigned long long sum = 0;
        for (int s = b; s < e; ++s) {
            int64_t ns, nb, off;
            if (gen_toy(A, s, &ns, &nb, &off)) sum += (unsigned long long)ns;
        }
        if (sum) atomicAdd(&events, sum);
    }
    G::acceptance(A, &per_cand);
    __syncthreads();
    float kept = per_cand * (float)kGenCand;
    const float many = (float)events / ((float)kGenPerWarp * (float)n_warps);   // kept per ticket that leaves kGenPerWarp
    int sub = 1;
    while (sub < kGenMaxSub && (kept < (float)kGenMinKept || 2.0f * kept <= fminf((float)kGenMostKept, many))) {
        sub *= 2;
        kept *= 2.0f;
    }
    const bool cut = kept >= (float)kGenMinKept && kept <= 2.0f * kGenCand;
    for (int round = 0; round < 2; ++round) {
        const bool split = round == 0 && cut;
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
        if ((int)threadIdx.x == nt - 1) {
            base[A.n_toys] = run[nt - 1];
            base[A.n_toys + 1] = sub;
        }
        break;
    }
}

// consts.cu's record is in place on the stream.  The workspace (ticket prefix,
// counter, status words) is allocated in stream order and given back after the
// kernel; without it (no memory, or more toys of few events than resident warps) a
// warp generates a toy alone, with the same events.
template <class G>
ipa_status launch_generator(GenArgs A, cudaStream_t s) {
    int dev = 0;
    cudaGetDevice(&dev);
    constexpr size_t smem = kGenWarps * sizeof(GenLists);
    static int occ[64] = {};
    int& per_sm = occ[dev & 63];
    if (per_sm == 0) {
        // with the record's tables the lists may exceed the default limit of shared memory
        ipa_status st = cuda_fail(cudaFuncSetAttribute(generate_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       (int)smem), "generator attribute");
        if (st != IPA_OK) return st;
        int v = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, generate_kernel<G>, kBlock, smem);
        per_sm = e == cudaSuccess && v >= 1 ? v : 1;
    }
    const int64_t most = (int64_t)sm_count() * per_sm;
    // Tickets at most, one per kBkgChunk background events among them.  A ticket accepts kept >=
    // kGenMinKept = 8 of a toy's n + 3 sqrt(n) + 8 events on average: n / 5 + 4 tickets.  With many
    // events it is larger: kept > kGenMostKept / 2, n / 40 + 2 tickets, or kept > events / (2
    // kGenPerWarp warps), 2 kGenPerWarp per warp, n / 128 and 7 a toy (3 sqrt(n) <= n / 16 + 36).  The
    // workspace follows what the events in work can need, not the buffers alone: 1000 events
    // into buffers of 2e8 took 90 us with n / 5 words to reset.
    const int64_t few = A.capacity / 5 + 4 * (int64_t)A.n_toys;
    const int64_t many = A.capacity / 40 + 2 * kGenPerWarp * kGenWarps * most + 7 * (int64_t)A.n_toys;
    const int64_t max_tickets = (few < many ? few : many) + A.capacity / kBkgChunk + A.n_toys + 1;
    const size_t words = (size_t)A.n_toys + 3 + (size_t)max_tickets;
    bool tickets = true;
    if constexpr (G::kBlockEvents > 0) {             // few events per toy, by the buffers' room
        tickets = A.capacity > (int64_t)G::kBlockEvents * A.n_toys;
        if (!tickets && A.n_toys <= most * kGenWarps) {
            const int64_t blocks = 8 * (int64_t)sm_count();
            generate_block_kernel<G><<<(unsigned)(A.n_toys < blocks ? A.n_toys : blocks), kBlock, 0, s>>>(A);
            return cuda_fail(cudaGetLastError(), "toygen kernel launch");
        }
    }
    void* ws = nullptr;
    if (tickets && pool_alloc(&ws, words * 8, s, "generator workspace") == IPA_OK) {
        ipa_status st = cuda_fail(cudaMemsetAsync(ws, 0, words * 8, s), "generator workspace reset");
        int64_t* base = static_cast<int64_t*>(ws);
        A.base = base;
        A.ticket = reinterpret_cast<unsigned long long*>(base + A.n_toys + 2);
        A.status = A.ticket + 1;
        if (st == IPA_OK) {
            gen_tickets_kernel<G><<<1, 1024, 0, s>>>(A, max_tickets, most * kGenWarps, base);
            const int64_t need = (max_tickets + kGenWarps - 1) / kGenWarps;
            generate_kernel<G><<<(unsigned)(need < most ? need : most), kBlock, smem, s>>>(A);
            st = cuda_fail(cudaGetLastError(), "toygen kernel launch");
        }
        pool_free(ws, s);
        return st;
    }
    cudaGetLastError();
    A.base = nullptr;
    const int64_t need = ((int64_t)A.n_toys + kGenWarps - 1) / kGenWarps;
    generate_kernel<G><<<(unsigned)(need < most ? need : most), kBlock, smem, s>>>(A);
    return cuda_fail(cudaGetLastError(), "toygen kernel launch");
}

}  // namespace ipa
