// Device code of the GB300 speculative coloring path (Algorithm 2 of the
// paper, "Iterative", Sec. 3.2, run in synchronous rounds).
//
// Fused pass k (k >= 2) over the worklist U_k, reading the colors C_k that
// round k's Phase 1 produced:
//   * Phase 2 of round k: v in U_k conflicts iff a neighbour w with
//     C_k[w] == C_k[v] precedes v ((prio[w], w) < (prio[v], v));
//   * Phase 1 of round k+1 for the conflicting v: first fit over the same
//     snapshot C_k (the smallest color > 0 no neighbour holds, Sec. 3.1).
// Both read adj(v) and C_k only, so one pass over adj(v) yields both; the
// two-phase form would read every adjacency twice.
//
// Double buffering: pass k reads X[k & 1] and writes X[(k + 1) & 1].  A
// vertex that settles writes its final color to both buffers, so no copy of
// the whole array is ever needed.  Round 1 colors every vertex 1 (all colors
// start at 0), so pass 1 needs no color reads: v conflicts iff some
// neighbour precedes it, and then its round-2 color is 2.
//
// Active neighbours.  A color word carries a flag bit once its vertex has
// settled (its color is final).  A vertex v still in U reads each neighbour's
// word anyway (the conflict test and first fit need this round's color), and
// a flagged neighbour is then folded into v's static mask (the colors held by
// settled neighbours, kept per vertex across rounds) and dropped: later rounds
// read only the neighbours that had not settled, plus v's static mask; first
// fit looks at static | this round's colors.  Rows of up to 121 entries drop a
// neighbour by clearing its bit; longer rows keep an active list, which pass k
// rewrites compacted into the other of two buffers, and a mask of the colors
// 1..256 (a first fit beyond 256 rescans the original row, every neighbour).
// The flag makes 16-bit state hold colors < 2^15: a larger color sets an
// overflow status and the host reruns with 32-bit state.
//
// Work is split into warp-sized tasks, binned by degree (L2 to L16) or by the
// current active length (S, M, H):
//   L2, L4 bins (degree <= 9 and <= 25, and s_max): the row is read from the
//     graph itself in 32-byte chunks by 2 or 4 lanes, with one bit per entry for
//     "not settled yet" in the worklist entry; no list is kept;
//   L8, L16 bins (longer rows of degree <= 57 and <= 121): likewise, by 8 or 16
//     lanes, the bits beside the static mask;
//   S bin (longer rows whose list has shrunk to s_max): 32 worklist entries per
//     task (down to 4 in the small rounds at the end), their lists walked as
//     one flat range;
//   M bin (other lists of s_max < length <= m_max <= 256): up to 16 worklist
//     entries per task, each list read by the whole warp in turn (colors 1..64
//     in registers);
//   H bin (length > m_max): one chunk of up to 1024 entries of one list per
//     task; a list of one chunk is decided by its warp, and the chunks of a
//     longer list OR their conflict flag and color windows into a per-vertex
//     record, write their survivors at offsets taken from an atomic counter,
//     and the warp that finishes the last chunk decides.
// Tasks are dealt to warps round-robin; after the round's split into tasks no
// block-wide barrier is taken inside a round.
//
// Priority: the round kernels are instantiated for index priority (the test
// is one compare) and for a priority array, whose (key, index) order round 2
// evaluates once per kept neighbour and stores in a bit mask (rows read from
// the graph) or in bit 31 of the active-list entry.  Loops: all rounds in one
// cooperative launch with a bounded grid barrier (optionally handing the last
// rounds to block 0), one launch per round, or a CUDA graph whose while node
// repeats a round kernel and a one-thread condition kernel.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gc {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBinS = 0, kBinM = 1, kBinH = 2;
constexpr int kPerLane = 8;                   // adjacency entries per lane in a hub chunk
constexpr int kSmallMaxLimit = 32;            // S bin: length <= 32
constexpr int kMedMaxLimit = 32 * kPerLane;   // M bin: length <= 256
constexpr int kHubSub = 32 * kPerLane;        // 256 entries: one sub-block of a hub chunk
constexpr int kChunk = 4 * kHubSub;           // 1024 entries per H-bin task
constexpr int kPass1Flat = 256;               // pass 1: longer open rows go to pass1_long_kernel
constexpr int kPass1LongBlocksPerSm = 8;      // pass 1, long rows: grid of 8 blocks per SM
#ifndef GC_FLAT_BATCHES
#define GC_FLAT_BATCHES 4
#endif
#ifndef GC_MIN_BLOCKS
#define GC_MIN_BLOCKS 4
#endif
#ifndef GC_MED_PER_TASK
#define GC_MED_PER_TASK 16
#endif

constexpr int kFlatBatches = GC_FLAT_BATCHES;  // flat tasks: batches in flight together
constexpr int kMedPerTask = GC_MED_PER_TASK;   // M-bin vertices per task
constexpr int kShortPerTaskMin = 4;            // S-bin vertices per task in a small round
constexpr int kMidSteps = 8;                  // L8, L16: steps of 32 / L vertices per task, at most

// L2 and L4 bins: degrees up to s_max whose row fits L chunks of eight entries
// wherever it starts (8 L - 7), and, with a priority array, whose state fits the
// worklist entry: a live and a precedence bit per entry and the colors 1..22.
constexpr int kKeyedBits = 21;
__host__ __device__ __forceinline__ int32_t tiny_limit(int L, int32_t s_max, bool keyed) {
    const int32_t fits = 8 * L - 7 < kKeyedBits || !keyed ? 8 * L - 7 : kKeyedBits;
    return s_max < fits ? s_max : fits;
}

// L8 and L16 bins: degrees above that (and up to m_max) whose row fits L chunks
// likewise.
__host__ __device__ __forceinline__ int32_t mid_limit(int L, int32_t s_max, int32_t m_max) {
    const int32_t most = 8 * L - 7 < m_max ? 8 * L - 7 : m_max;
    return most > s_max ? most : s_max;
}
constexpr int kMinBlocks = GC_MIN_BLOCKS;      // round kernels: blocks per SM the registers allow
constexpr int kWarpsPerBlockMax = 8;          // blocks of <= 256 threads

// Status codes shared with gc.h (kept numerically equal), and one internal.
constexpr int kStatusOk = 0;
constexpr int kStatusMaxRounds = -4;
constexpr int kStatusTimeout = -5;
constexpr int kStatusColorOverflow = -100;    // 16-bit state too narrow: rerun with 32-bit

// A grid barrier gives up after this long (globaltimer ns) or this many polls.
constexpr unsigned long long kBarrierTimeoutNs = 4000000000ull;
constexpr unsigned kBarrierMaxPolls = 1u << 26;

// Settled flag and color field of a color word.
template <typename T> struct Word;
template <> struct Word<uint16_t> { static constexpr uint32_t kFlag = 0x8000u; };
template <> struct Word<int32_t> { static constexpr uint32_t kFlag = 0x80000000u; };

template <typename T>
__device__ __forceinline__ uint32_t word_raw(T x) {
    return sizeof(T) == 2 ? (uint32_t)(uint16_t)x : (uint32_t)x;
}
template <typename T>
__device__ __forceinline__ uint32_t word_color(T x) { return word_raw(x) & (Word<T>::kFlag - 1u); }
template <typename T>
__device__ __forceinline__ bool word_settled(T x) { return (word_raw(x) & Word<T>::kFlag) != 0u; }

struct Stats {
    int max_degree;
    int bad;                      // rowptr[0] != 0 or a negative degree
    int nnz;                      // rowptr[n]
    unsigned defer;               // vertices with degree > kPass1Flat
    unsigned cap[3];              // vertices with degree >= 1, > tiny_limit(4), > m_max
    unsigned over2, over8, over16;  // with degree > tiny_limit(2), > mid_limit(8), > mid_limit(16)
    unsigned long long hub_chunks;  // sum over degree > m_max of ceil(degree / kChunk)
};

// One round's worklist counters.  Every warp appends through them, so each
// sits on its own 128-byte line (its own L2 slice): on one line, the atomics
// of all bins queued at one slice, which then served a quarter more requests
// than any other.  A hub's two counters (its worklist position and its first
// chunk) share one 64-bit word, taken with one atomic.
struct RoundCounts {
    alignas(128) unsigned long long tiny;  // |U_k in L2| (bits 0..31) | |U_k in L4| (bits 32..63)
    unsigned overflow;                     // round k - 1 chose a color too wide for the state
    alignas(128) unsigned long long mid;   // |U_k in L8| (bits 0..31) | |U_k in L16| (bits 32..63)
    alignas(128) unsigned s;               // |U_k in S|
    alignas(128) unsigned m;               // |U_k in M|
    alignas(128) unsigned long long hc;    // |U_k in H| (bits 0..31) | chunks of U_k in H (bits 32..63)
    alignas(128) unsigned vol;             // active entries round k reads
};

// Two 32-bit counts in one 64-bit word.
__host__ __device__ __forceinline__ unsigned low_count(unsigned long long x) { return (unsigned)x; }
__host__ __device__ __forceinline__ unsigned high_count(unsigned long long x) { return (unsigned)(x >> 32); }
__host__ __device__ __forceinline__ unsigned long long pair_count(unsigned low, unsigned high) {
    return ((unsigned long long)high << 32) | (unsigned long long)low;
}
__host__ __device__ __forceinline__ unsigned hub_count(unsigned long long hc) { return (unsigned)hc; }
__host__ __device__ __forceinline__ unsigned hub_chunks(unsigned long long hc) { return (unsigned)(hc >> 32); }

// The append counters, the two barrier words and the result words sit on
// separate 128-byte lines, so that blocks polling the barrier do not slow
// down the atomics of blocks still working.
struct RoundState {
    RoundCounts rc[3];     // [k % 3]: the counts of U_k
    alignas(128) unsigned defer_cnt;  // pass 1: rows left to pass1_long_kernel
    alignas(128) unsigned task_next[3];  // [k % 3]: tasks of round k claimed so far (beyond the first two per warp)
    alignas(128) unsigned bar_count;  // blocks that have reached a barrier, over all barriers
    alignas(128) int status;
    int rounds;
    int max_color;
    int graph_round;       // loop mode 2: the round the graph's next iteration runs
};

// Per H-bin vertex of the current round (indexed by its worklist position).
struct HubRecord {
    unsigned mask[8];      // colors 1..256 seen by any chunk this round
    unsigned stat[8];      // colors 1..256 of neighbours found settled this round
    unsigned conflict;
    unsigned done;         // chunks finished
    unsigned kept;         // active entries kept for the next round
    unsigned pad[13];
};

template <typename T>
struct Params {
    const int32_t* __restrict__ rowptr;
    const int32_t* __restrict__ colidx;
    const uint32_t* __restrict__ prio;  // NULL = index priority
    int32_t n;
    int32_t nnz;                        // entries of colidx
    int32_t s_max, m_max;               // length bin limits
    int32_t lim2, lim4, lim8, lim16;    // degree limits of the L2, L4, L8 and L16 bins
    int32_t max_rounds;
    int32_t tail_volume;                // rounds reading <= this many entries run in block 0 alone (< 0: never)
    uint32_t barrier_polls;             // the grid barrier gives up after this many polls
    uint32_t color_limit;               // a color >= this overflows (16-bit state)
    T* X0;
    T* X1;
    int32_t* colors_out;
    int32_t* settle_round;              // NULL, or receives the round in which each vertex settled
    int32_t* act0;                      // active lists (row starts as in colidx)
    int32_t* act1;
    uint32_t* stat;                     // static masks, 8 words per vertex
    // worklists per parity (A: even k, B: odd k): L2 and L4 entries {vertex, row
    // start, live entries, static mask}; L8, L16, S, M, H entries {vertex, row start,
    // active length (L8, L16: degree), degree}, first chunk of each H entry,
    // owner position of each chunk
    int4* L2A; int4* L4A; int4* L8A; int4* L16A; int4* SA; int4* MA; int4* HA; int32_t* HcA; int32_t* OA;
    int4* L2B; int4* L4B; int4* L8B; int4* L16B; int4* SB; int4* MB; int4* HB; int32_t* HcB; int32_t* OB;
    int32_t* defer;                     // pass 1: long rows left open
    HubRecord* hubs;
    RoundState* st;
    int32_t* round_sizes;               // device telemetry, round_sizes[k-1] = |U_k|
    unsigned long long* round_vol;      // device telemetry, round_vol[k-1] = entries round k reads
    unsigned long long* round_ns;       // NULL, or device telemetry: round_ns[k-1] = %globaltimer when
                                        // round k's pass starts (persistent launch; round_cap + 1 entries)
    int32_t round_cap;
};

// ------------------------------------------------------------ helpers

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

// L2 eviction policies: adjacency is streamed and should not push the color
// arrays (gathered at random) out of L2.
__device__ __forceinline__ uint64_t policy_evict_first() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

#ifndef GC_L1_COLORS
#define GC_L1_COLORS 1
#endif

// Adjacency / active-list entry.  colidx is read-only for the whole call;
// an active list is written in one round and read in the next.  Rounds are
// separated by kernel boundaries or by grid_barrier, whose fences make
// earlier rounds' writes visible to cached loads after it (the ordering a
// grid-wide synchronisation gives), so these loads may use L1.
__device__ __forceinline__ int32_t ld_row(const int32_t* a, uint64_t pol) {
    int32_t r;
#if GC_L1_COLORS
    asm volatile("ld.global.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(r) : "l"(a), "l"(pol));
#else
    asm volatile("ld.global.cg.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(r) : "l"(a), "l"(pol));
#endif
    return r;
}
__device__ __forceinline__ int32_t ld_adj(const int32_t* a, uint64_t pol) {
    int32_t r;
    asm volatile("ld.global.nc.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(r) : "l"(a), "l"(pol));
    return r;
}

// Color word: written in earlier rounds (visible after the round boundary,
// as above) and kept in L2 (evict_last); the few high-degree vertices that
// most gathers hit stay in each SM's L1.  Within a round a word may gain its
// settled flag while others read it; a copy without the flag is still the
// right color, and the flag is seen a round later.
__device__ __forceinline__ uint16_t ld_color(const uint16_t* a, uint64_t pol) {
    uint16_t r;
#if GC_L1_COLORS
    asm volatile("ld.global.L2::cache_hint.u16 %0, [%1], %2;" : "=h"(r) : "l"(a), "l"(pol));
#else
    asm volatile("ld.global.cg.L2::cache_hint.u16 %0, [%1], %2;" : "=h"(r) : "l"(a), "l"(pol));
#endif
    return r;
}
__device__ __forceinline__ int32_t ld_color(const int32_t* a, uint64_t pol) {
    int32_t r;
#if GC_L1_COLORS
    asm volatile("ld.global.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(r) : "l"(a), "l"(pol));
#else
    asm volatile("ld.global.cg.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(r) : "l"(a), "l"(pol));
#endif
    return r;
}

// With a priority array, active lists written from round 2 on carry, in bit
// 31 of each entry (ids are below 2^31), whether that neighbour precedes the
// list's vertex.  The order never changes, so it is computed once (round 2)
// and later rounds test a bit instead of gathering two priority keys per
// equally colored neighbour.  Under index priority the test is one compare
// and the lists carry plain ids.
constexpr uint32_t kPrecBit = 0x80000000u;
__device__ __forceinline__ int32_t entry_id(int32_t x) { return x & 0x7fffffff; }

// w precedes v: (prio[w], w) < (prio[v], v); pv = prio[v] (ignored if no prio).
__device__ __forceinline__ bool precedes(const uint32_t* __restrict__ prio, int32_t w, int32_t v,
                                         uint32_t pv) {
    if (prio) {
        const uint32_t pw = __ldg(prio + w);
        if (pw != pv) return pw < pv;
    }
    return w < v;
}

// Append a worklist entry (if flag) with one atomic per warp.  All lanes call it.
__device__ __forceinline__ void warp_append(bool flag, int4 e, int4* list, unsigned* cnt) {
    const unsigned ballot = __ballot_sync(kFull, flag);
    if (ballot == 0) return;
    const unsigned lane = lane_id();
    const int leader = __ffs(ballot) - 1;
    unsigned base = 0;
    if ((int)lane == leader) base = atomicAdd(cnt, (unsigned)__popc(ballot));
    base = __shfl_sync(kFull, base, leader);
    if (flag) list[base + __popc(ballot & ((1u << lane) - 1u))] = e;
}

// The same with a counter in the bits from SHIFT (0 or 32) on of a 64-bit word.
template <int SHIFT>
__device__ __forceinline__ void warp_append_pair(bool flag, int4 e, int4* list, unsigned long long* cnt) {
    const unsigned ballot = __ballot_sync(kFull, flag);
    if (ballot == 0) return;
    const unsigned lane = lane_id();
    unsigned base = 0;
    if (lane == 0) base = (unsigned)(atomicAdd(cnt, (unsigned long long)__popc(ballot) << SHIFT) >> SHIFT);
    base = __shfl_sync(kFull, base, 0);
    if (flag) list[base + __popc(ballot & ((1u << lane) - 1u))] = e;
}

// Where the next round's worklists go.
struct NextLists {
    int4* L2; int4* L4; int4* L8; int4* L16; int4* S; int4* M; int4* H; int32_t* Hc; int32_t* O;
    RoundCounts* cnt;  // the next round's counts
    int32_t s_max, m_max;
};

__device__ __forceinline__ int bin_of(int32_t len, int32_t s_max, int32_t m_max) {
    return len <= s_max ? kBinS : (len <= m_max ? kBinM : kBinH);
}

// Append H-bin entry e (lane 0's copy) to the next round and hand it its
// chunks.  Called by all lanes of a warp.
__device__ __forceinline__ void warp_append_hub(const NextLists& nl, int4 e) {
    const unsigned nch = (unsigned)(e.z + kChunk - 1) / kChunk;
    unsigned pos = 0, c0 = 0;
    if (lane_id() == 0) {
        const unsigned long long old = atomicAdd(&nl.cnt->hc, ((unsigned long long)nch << 32) | 1ull);
        pos = hub_count(old);
        c0 = hub_chunks(old);
        nl.H[pos] = e;
        nl.Hc[pos] = (int32_t)c0;
    }
    pos = __shfl_sync(kFull, pos, 0);
    c0 = __shfl_sync(kFull, c0, 0);
    for (unsigned j = lane_id(); j < nch; j += 32) nl.O[c0 + j] = (int32_t)pos;
}

// Append the H-bin entries of the lanes whose flag is set, with one atomic for
// all of them (their chunks get consecutive ranges).  Called by all lanes.
__device__ __forceinline__ void warp_append_hubs(const NextLists& nl, bool flag, int4 e) {
    const unsigned ballot = __ballot_sync(kFull, flag);
    if (ballot == 0) return;
    const unsigned lane = lane_id();
    const unsigned nch = flag ? (unsigned)(e.z + kChunk - 1) / kChunk : 0u;
    unsigned incl = nch;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned x = __shfl_up_sync(kFull, incl, o);
        if ((int)lane >= o) incl += x;
    }
    const unsigned total = __shfl_sync(kFull, incl, 31);
    unsigned long long old = 0;
    if (lane == 0) old = atomicAdd(&nl.cnt->hc, ((unsigned long long)total << 32) | (unsigned long long)__popc(ballot));
    old = __shfl_sync(kFull, old, 0);
    if (flag) {
        const unsigned pos = hub_count(old) + (unsigned)__popc(ballot & ((1u << lane) - 1u));
        const unsigned c0 = hub_chunks(old) + incl - nch;
        nl.H[pos] = e;
        nl.Hc[pos] = (int32_t)c0;
        for (unsigned j = 0; j < nch; ++j) nl.O[c0 + j] = (int32_t)pos;
    }
}

// The lowest d bits (0 <= d <= 32).
__device__ __forceinline__ uint32_t low_bits(int32_t d) { return d >= 32 ? 0xffffffffu : (1u << d) - 1u; }

// Append one entry held by lane 0 (any bin).  Called by all lanes of a warp.
__device__ __forceinline__ void warp_append_one(const NextLists& nl, int4 e) {
    const int bin = bin_of(e.z, nl.s_max, nl.m_max);
    if (bin == kBinH) {
        warp_append_hub(nl, e);
    } else if (lane_id() == 0) {
        int4* list = bin == kBinM ? nl.M : nl.S;
        list[atomicAdd(bin == kBinM ? &nl.cnt->m : &nl.cnt->s, 1u)] = e;
    }
}

// x << s with shifts of 32 and more (or "negative" ones) giving 0.
__device__ __forceinline__ uint32_t shl_clamp(uint32_t x, uint32_t s) {
    uint32_t r;
    asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
    return r;
}

// Bits of colors base+1 .. base+256 seen by one lane.
struct Mask256 {
    uint64_t w0, w1, w2, w3;
    __device__ __forceinline__ void clear() { w0 = w1 = w2 = w3 = 0; }
    // idx = color - 1 - base; anything outside [0, 256) is ignored
    __device__ __forceinline__ void set(unsigned idx) {
        if (idx < 256u) {
            const uint64_t bit = 1ull << (idx & 63u);
            const unsigned q = idx >> 6;
            w0 |= (q == 0u) ? bit : 0ull;
            w1 |= (q == 1u) ? bit : 0ull;
            w2 |= (q == 2u) ? bit : 0ull;
            w3 |= (q == 3u) ? bit : 0ull;
        }
    }
    // OR over the warp; every lane receives word `lane & 7` of the result.
    __device__ __forceinline__ uint32_t warp_reduce_word() const {
        const uint32_t r0 = __reduce_or_sync(kFull, (uint32_t)w0);
        const uint32_t r1 = __reduce_or_sync(kFull, (uint32_t)(w0 >> 32));
        const uint32_t r2 = __reduce_or_sync(kFull, (uint32_t)w1);
        const uint32_t r3 = __reduce_or_sync(kFull, (uint32_t)(w1 >> 32));
        const uint32_t r4 = __reduce_or_sync(kFull, (uint32_t)w2);
        const uint32_t r5 = __reduce_or_sync(kFull, (uint32_t)(w2 >> 32));
        const uint32_t r6 = __reduce_or_sync(kFull, (uint32_t)w3);
        const uint32_t r7 = __reduce_or_sync(kFull, (uint32_t)(w3 >> 32));
        const unsigned q = lane_id() & 7u;
        uint32_t r = r0;
        r = q == 1u ? r1 : r;
        r = q == 2u ? r2 : r;
        r = q == 3u ? r3 : r;
        r = q == 4u ? r4 : r;
        r = q == 5u ? r5 : r;
        r = q == 6u ? r6 : r;
        r = q == 7u ? r7 : r;
        return r;
    }
};

// First clear bit of the 256-bit window whose word q sits in lanes with
// (lane & 7) == q; -1 if all set.  All lanes call it and get the same value.
__device__ __forceinline__ int window_first_clear(uint32_t word) {
    const unsigned notfull = __ballot_sync(kFull, lane_id() < 8u && word != 0xffffffffu);
    if (notfull == 0) return -1;
    const int q = __ffs(notfull) - 1;
    const uint32_t wq = __shfl_sync(kFull, word, q);
    return q * 32 + __ffs(~wq) - 1;
}

// First fit beyond the first window: rescan v's whole original row (settled
// neighbours were dropped from the active list) for windows base+1 .. until
// one has a free color.  Terminates: a full window of 256 colors needs 256
// more neighbours, and first fit never exceeds degree + 1.
template <typename T>
__device__ __forceinline__ unsigned rescan_first_fit(const int32_t* __restrict__ rowptr,
                                                     const int32_t* __restrict__ colidx, const T* Xc,
                                                     int32_t v) {
    const int32_t b = __ldg(rowptr + v), e = __ldg(rowptr + v + 1);
    for (unsigned base = 256u;; base += 256u) {
        Mask256 m;
        m.clear();
        for (int32_t i = b + (int32_t)lane_id(); i < e; i += 32)
            m.set(word_color(__ldcg(Xc + __ldg(colidx + i))) - 1u - base);
        const int ff = window_first_clear(m.warp_reduce_word());
        if (ff >= 0) return base + (unsigned)ff + 1u;
    }
}

// --------------------------------------------------- bounded grid barrier

__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// All blocks of a cooperative launch meet here, for the `passed`-th time
// (from 0).  Returns false (and sets status = timeout) if the wait gave up;
// the caller then leaves the loop.  Every block adds one to a count that is
// never reset and waits until all of them have: one round trip to L2 to
// arrive and one to see the last arrival.  (With a reset count, a generation
// word and the status read behind them, a round of nearly no work took 6.4 us
// of which this barrier was most; now 4.5 us.)
__device__ __forceinline__ bool grid_barrier(RoundState* st, unsigned max_polls, unsigned passed) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned all = gridDim.x * (passed + 1u);  // counts wrap around alike
        fence_gpu();
        volatile unsigned* count = &st->bar_count;
        if (atomicAdd(&st->bar_count, 1u) + 1u != all) {
            const unsigned long long t0 = globaltimer_ns();
            unsigned polls = 0;
            while ((int)(*count - all) < 0) {
                if (++polls > 4u) __nanosleep(polls < 32u ? 32 : 128);
                if (polls >= max_polls || globaltimer_ns() - t0 > kBarrierTimeoutNs ||
                    ((polls & 255u) == 0u && *((volatile int*)&st->status) == kStatusTimeout)) {
                    atomicExch(&st->status, kStatusTimeout);
                    ok = 0;
                    break;
                }
            }
        }
        fence_gpu();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

__device__ __forceinline__ void fold_max_color(RoundState* st, int maxc) {
    const int m = __reduce_max_sync(kFull, maxc);
    if (lane_id() == 0 && m > 0) atomicMax(&st->max_color, m);
}

// Add a warp's share of round r's read volume to the round counter
// (rc[r % 3].vol) and to the telemetry (round_vol[r-1]).
__device__ __forceinline__ void fold_volume(RoundState* st, unsigned long long* round_vol, int32_t cap, int r,
                                            unsigned vol) {
    const unsigned s = __reduce_add_sync(kFull, vol);
    if (lane_id() == 0 && s) {
        atomicAdd(&st->rc[r % 3].vol, s);
        if (r - 1 < cap) atomicAdd(&round_vol[r - 1], (unsigned long long)s);
    }
}

// ------------------------------------------------------------ setup scan

// Degree statistics: max degree, list capacities, hub chunks, rowptr checks.
__global__ void stats_kernel(const int32_t* __restrict__ rowptr, int32_t n, int32_t s_max,
                             int32_t m_max, bool keyed, Stats* s) {
    int mx = 0, bad = 0;
    unsigned c0 = 0, c1 = 0, c2 = 0, df = 0, o2 = 0, o8 = 0, o16 = 0;
    unsigned long long ch = 0;
    const int32_t tiny2 = tiny_limit(2, s_max, keyed), tiny4 = tiny_limit(4, s_max, keyed);
    const int32_t mid8 = mid_limit(8, s_max, m_max), mid16 = mid_limit(16, s_max, m_max);
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
         v += (int64_t)gridDim.x * blockDim.x) {
        const int32_t d = __ldg(rowptr + v + 1) - __ldg(rowptr + v);
        if (d < 0) { bad = 1; continue; }
        mx = max(mx, d);
        c0 += d >= 1;
        c1 += d > tiny4;
        o2 += d > tiny2;
        c2 += d > m_max;
        o8 += d > mid8;
        o16 += d > mid16;
        df += d > kPass1Flat;
        if (d > m_max) ch += (unsigned long long)((d + kChunk - 1) / kChunk);
    }
    mx = __reduce_max_sync(kFull, mx);
    bad = __reduce_or_sync(kFull, (unsigned)bad);
    c0 = __reduce_add_sync(kFull, c0);
    c1 = __reduce_add_sync(kFull, c1);
    c2 = __reduce_add_sync(kFull, c2);
    df = __reduce_add_sync(kFull, df);
    o2 = __reduce_add_sync(kFull, o2);
    o8 = __reduce_add_sync(kFull, o8);
    o16 = __reduce_add_sync(kFull, o16);
    if (lane_id() == 0) {
        atomicMax(&s->max_degree, mx);
        if (bad) s->bad = 1;
        if (c0) atomicAdd(&s->cap[0], c0);
        if (c1) atomicAdd(&s->cap[1], c1);
        if (c2) atomicAdd(&s->cap[2], c2);
        if (df) atomicAdd(&s->defer, df);
        if (o2) atomicAdd(&s->over2, o2);
        if (o8) atomicAdd(&s->over8, o8);
        if (o16) atomicAdd(&s->over16, o16);
    }
    for (int o = 16; o > 0; o >>= 1) ch += __shfl_xor_sync(kFull, ch, o);
    if (lane_id() == 0 && ch) atomicAdd(&s->hub_chunks, ch);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (__ldg(rowptr) != 0) s->bad = 1;
        s->nnz = __ldg(rowptr + n);
    }
}

// ------------------------------------------------------------- pass 1

// Outcome of round 1 for v: C_2[v] = 2 if it conflicts (then it joins U_2),
// else v keeps color 1 for good (flagged in both buffers).
template <typename T>
__device__ __forceinline__ void pass1_write(const Params<T>& p, int32_t v, bool conflict, int& maxc) {
    if (conflict) {
        p.X0[v] = (T)2;
    } else {
        const T one = (T)(1u | Word<T>::kFlag);
        p.X0[v] = one;
        p.X1[v] = one;
        p.colors_out[v] = 1;
        if (p.settle_round) p.settle_round[v] = 1;
        maxc = 1;
    }
}

template <typename T>
__device__ __forceinline__ NextLists pass1_next(const Params<T>& p) {
    NextLists nl;
    nl.L2 = p.L2A; nl.L4 = p.L4A; nl.L8 = p.L8A; nl.L16 = p.L16A;
    nl.S = p.SA; nl.M = p.MA; nl.H = p.HA; nl.Hc = p.HcA; nl.O = p.OA;
    nl.cnt = &p.st->rc[2];
    nl.s_max = p.s_max;
    nl.m_max = p.m_max;
    return nl;
}

// Eight consecutive entries of colidx from index a on (a multiple of eight
// counted from the 32-byte boundary at or below colidx), with one 32-byte
// load; where that would reach outside the array, entry by entry.
__device__ __forceinline__ void load_chunk(const int32_t* __restrict__ colidx, int32_t nnz, int32_t a, uint64_t pol,
                                           int32_t (&w)[8]) {
    if (a >= 0 && a <= nnz - 8) {
        asm volatile("ld.global.nc.L2::cache_hint.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8], %9;"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                     : "l"(colidx + a), "l"(pol));
    } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) w[u] = a + u >= 0 && a + u < nnz ? __ldg(colidx + a + u) : 0;
    }
}

// Whether one of the chunk's entries at positions [U0, U1) that `in` marks precedes v.
template <int U0, int U1>
__device__ __forceinline__ bool chunk_precedes(const uint32_t* __restrict__ prio, const int32_t (&w)[8], uint32_t in,
                                               int32_t v, uint32_t pv) {
    bool hit = false;
    if (prio) {
        uint32_t pw[U1 - U0];
#pragma unroll
        for (int u = U0; u < U1; ++u) pw[u - U0] = (in >> u) & 1u ? __ldg(prio + w[u]) : 0xffffffffu;
#pragma unroll
        for (int u = U0; u < U1; ++u)
            hit |= ((in >> u) & 1u) && (pw[u - U0] < pv || (pw[u - U0] == pv && w[u] < v));
    } else {
#pragma unroll
        for (int u = U0; u < U1; ++u) hit |= ((in >> u) & 1u) && w[u] < v;
    }
    return hit;
}

// The positions of a chunk at offset off of a row of d entries that lie in the row.
__device__ __forceinline__ uint32_t chunk_in_row(int32_t off, int32_t d) {
    return low_bits(max(0, min(8, d - off))) & (off < 0 ? 0xffu << -off : 0xffu);
}

// Round 1 over vertices [v_begin, v_end) (the host may launch it per range as
// the input arrives): a vertex conflicts iff a neighbour precedes it, and one
// such neighbour decides that, so a row is read only as far as needed.  A
// block takes 256 PER vertices at a time.  Every thread reads the first
// 32-byte chunk of its rows (all of it under index priority; half the chunk at a
// time when a key has to be gathered for each entry).  Rows that this
// leaves open, local minima for the most part, are read on by four lanes each
// from a list in shared memory, or, when longer than kPass1Flat, go to
// pass1_long_kernel.  The block appends its entries with one atomic per counter.
//
// Bound: one 32-byte sector of colidx per vertex, and its row start, buffers and
// worklist entry.  Reading every row to its end as one flat range took 0.71 ms
// for R-MAT-B of 2^24 vertices (now 0.38; both with the setup scan, 0.07 of it)
// and 0.24 for R-MAT-ER of 2^22 (now 0.10).
//
// PER vertices a thread: 4, or 1 for a range too small to give every SM a block
// of 1,024.
template <typename T, int PER>
__global__ void __launch_bounds__(256, 4) pass1_kernel(Params<T> p, int32_t v_begin, int32_t v_end) {
    constexpr int kPass1Per = PER, kPass1Block = 256 * PER;
    constexpr int kBins = 6;                // L2, L4, L8, L16, M entries; long rows left open
    __shared__ int32_t s_b[kPass1Block], s_d[kPass1Block];
    __shared__ uint16_t s_open[kPass1Block];  // vertices of this block whose first chunk left them open
    __shared__ uint8_t s_hit[kPass1Block];
    __shared__ unsigned s_nopen, s_cnt[kBins], s_base[kBins];
    __shared__ unsigned long long s_hub, s_hub_base;
    const NextLists nl = pass1_next(p);
    const uint64_t pol = policy_evict_first();
    const uint32_t mis = (uint32_t)((uintptr_t)p.colidx >> 2) & 7u;
    const unsigned tid = threadIdx.x, lane = lane_id();
    const unsigned below = (1u << lane) - 1u;
    int maxc = 0;
    unsigned vol = 0;
    for (int64_t first = (int64_t)v_begin + (int64_t)blockIdx.x * kPass1Block; first < v_end;
         first += (int64_t)gridDim.x * kPass1Block) {
        if (tid < kBins) s_cnt[tid] = 0u;
        if (tid == kBins) s_nopen = 0u;
        if (tid == kBins + 1) s_hub = 0ull;
        __syncthreads();
        int32_t b[kPass1Per], d[kPass1Per];
        unsigned hits = 0u, opens = 0u;  // bit i: this thread's vertex i
#pragma unroll
        for (int i = 0; i < kPass1Per; ++i) {
            const int64_t vv = first + i * 256 + tid;
            b[i] = vv < v_end ? __ldg(p.rowptr + vv) : 0;
            d[i] = vv < v_end ? __ldg(p.rowptr + vv + 1) - b[i] : 0;
        }
#pragma unroll
        for (int i = 0; i < kPass1Per; ++i) {
            const int32_t v = (int32_t)(first + i * 256 + tid);
            const int32_t off = -(int32_t)(((uint32_t)b[i] + mis) & 7u);
            bool hit = false;
            if (d[i] > 0) {
                int32_t w[8];
                load_chunk(p.colidx, p.nnz, b[i] + off, pol, w);
                const uint32_t in = chunk_in_row(off, d[i]);
                const uint32_t pv = p.prio ? __ldg(p.prio + v) : 0u;
                hit = chunk_precedes<4, 8>(p.prio, w, in, v, pv);
                if (!hit) hit = chunk_precedes<0, 4>(p.prio, w, in, v, pv);
            }
            const bool open = !hit && off + 8 < d[i];
            hits |= hit ? 1u << i : 0u;
            opens |= open ? 1u << i : 0u;
            const unsigned ball = __ballot_sync(kFull, open && d[i] <= kPass1Flat);
            if (ball) {
                unsigned at = 0;
                if (lane == 0) at = atomicAdd(&s_nopen, (unsigned)__popc(ball));
                at = __shfl_sync(kFull, at, 0) + __popc(ball & below);
                if ((ball >> lane) & 1u) {
                    const unsigned slot = i * 256 + tid;
                    s_open[at] = (uint16_t)slot;
                    s_b[slot] = b[i];
                    s_d[slot] = d[i];
                }
            }
        }
        __syncthreads();
        // open rows: four lanes each, 64 side by side
        for (unsigned at = tid >> 2; at < ((s_nopen + 7u) & ~7u); at += 64u) {
            const bool on = at < s_nopen;
            const unsigned slot = on ? s_open[at] : 0u;
            const int32_t v = (int32_t)(first + slot), ob = on ? s_b[slot] : 0, od = on ? s_d[slot] : 0;
            const uint32_t pv = p.prio && on ? __ldg(p.prio + v) : 0u;
            bool hit = false;
            int32_t off = 8 + 8 * (int32_t)(lane & 3u) - (int32_t)(((uint32_t)ob + mis) & 7u);
            for (; off < od && !hit; off += 32) {
                int32_t w[8];
                load_chunk(p.colidx, p.nnz, ob + off, pol, w);
                hit = chunk_precedes<0, 8>(p.prio, w, chunk_in_row(off, od), v, pv);
            }
            const unsigned any = __ballot_sync(kFull, hit) >> (lane & ~3u) & 15u;
            if (on && (lane & 3u) == 0u) s_hit[slot] = any != 0u;
        }
        __syncthreads();
        // outcome, and this block's share of every worklist
        int cls[kPass1Per];
        unsigned at[kPass1Per];
        unsigned long long hub_at[kPass1Per];
#pragma unroll
        for (int i = 0; i < kPass1Per; ++i) {
            const int64_t vv = first + i * 256 + tid;
            const bool later = (opens >> i & 1u) && d[i] > kPass1Flat;  // decided by pass1_long_kernel
            const bool hit = (hits >> i & 1u) || ((opens >> i & 1u) && !later && s_hit[i * 256 + tid]);
            cls[i] = -1;
            if (vv < v_end) {
                if (!later) {
                    pass1_write(p, (int32_t)vv, hit, maxc);
                    if (hit) vol += (unsigned)d[i];
                }
                if (later) cls[i] = 5;
                else if (hit) cls[i] = d[i] <= p.lim8 ? (d[i] <= p.lim2 ? 0 : (d[i] <= p.lim4 ? 1 : 2))
                                                      : (d[i] <= p.lim16 ? 3 : (d[i] <= p.m_max ? 4 : 6));
            }
            at[i] = 0u;
#pragma unroll
            for (int c = 0; c < kBins; ++c) {
                const unsigned bal = __ballot_sync(kFull, cls[i] == c);
                if (bal == 0u) continue;
                unsigned base = 0;
                if (lane == 0) base = atomicAdd(&s_cnt[c], (unsigned)__popc(bal));
                base = __shfl_sync(kFull, base, 0);
                if (cls[i] == c) at[i] = base + __popc(bal & below);
            }
            hub_at[i] = 0ull;
            const unsigned hubs = __ballot_sync(kFull, cls[i] == 6);
            if (hubs) {
                const unsigned chunks = cls[i] == 6 ? (unsigned)(d[i] + kChunk - 1) / kChunk : 0u;
                unsigned upto = chunks;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned x = __shfl_up_sync(kFull, upto, o);
                    if ((int)lane >= o) upto += x;
                }
                unsigned long long base = 0ull;
                if (lane == 31u) base = atomicAdd(&s_hub, pair_count(__popc(hubs), upto));
                hub_at[i] = __shfl_sync(kFull, base, 31) + pair_count(__popc(hubs & below), upto - chunks);
            }
        }
        __syncthreads();
        if (tid == 0 && (s_cnt[0] | s_cnt[1])) {
            const unsigned long long x = atomicAdd(&nl.cnt->tiny, pair_count(s_cnt[0], s_cnt[1]));
            s_base[0] = low_count(x);
            s_base[1] = high_count(x);
        }
        if (tid == 32 && (s_cnt[2] | s_cnt[3])) {
            const unsigned long long x = atomicAdd(&nl.cnt->mid, pair_count(s_cnt[2], s_cnt[3]));
            s_base[2] = low_count(x);
            s_base[3] = high_count(x);
        }
        if (tid == 64 && s_cnt[4]) s_base[4] = atomicAdd(&nl.cnt->m, s_cnt[4]);
        if (tid == 96 && s_cnt[5]) s_base[5] = atomicAdd(&p.st->defer_cnt, s_cnt[5]);
        if (tid == 128 && s_hub) s_hub_base = atomicAdd(&nl.cnt->hc, s_hub);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kPass1Per; ++i) {
            const int32_t v = (int32_t)(first + i * 256 + tid);
            if (cls[i] == 6) {
                // (both halves of the pair stay below 2^32: no carry)
                const unsigned long long x = s_hub_base + hub_at[i];
                const unsigned pos = hub_count(x), c0 = hub_chunks(x);
                nl.H[pos] = make_int4(v, b[i], d[i], d[i]);
                nl.Hc[pos] = (int32_t)c0;
                for (unsigned j = 0; j < (unsigned)(d[i] + kChunk - 1) / kChunk; ++j) nl.O[c0 + j] = (int32_t)pos;
            } else if (cls[i] == 5) {
                p.defer[s_base[5] + at[i]] = v;
            } else if (cls[i] >= 0) {
                int4* const list = cls[i] == 0 ? p.L2A
                                               : (cls[i] == 1 ? p.L4A : (cls[i] == 2 ? p.L8A : (cls[i] == 3 ? p.L16A : p.MA)));
                // an L2 or L4 entry starts with all of its row live and no static mask
                list[s_base[cls[i]] + at[i]] =
                    cls[i] <= 1 ? make_int4(v, b[i], (int32_t)low_bits(d[i]), 0) : make_int4(v, b[i], d[i], d[i]);
            }
        }
        __syncthreads();
    }
    fold_max_color(p.st, maxc);
    fold_volume(p.st, p.round_vol, p.round_cap, 2, vol);
}

// Round 1 for rows longer than kPass1Flat whose first chunk decided nothing: a
// warp takes up to 32 of them (one per lane; fewer when there are not many, so
// that every warp has some),
// reads them one after another, 128 entries per step, stopping at the first
// preceding neighbour, and appends the conflicting ones (all H bin: longer
// than kPass1Flat >= m_max) with one atomic.
template <typename T>
__global__ void __launch_bounds__(256) pass1_long_kernel(Params<T> p) {
    const unsigned lane = lane_id();
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t W = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const unsigned nd = __ldcg(&p.st->defer_cnt);
    const NextLists nl = pass1_next(p);
    const uint64_t pol_adj = policy_evict_first();
    int maxc = 0;
    unsigned vol = 0;
    const int64_t R = max((int64_t)1, min((int64_t)32, ((int64_t)nd + W - 1) / W));  // rows per warp
    for (int64_t t0 = gw * R; t0 < nd; t0 += W * R) {
        const int64_t i = t0 + lane;
        const bool valid = lane < R && i < nd;
        const int32_t v = valid ? __ldcg(p.defer + i) : 0;
        const int32_t b = valid ? __ldg(p.rowptr + v) : 0, e = valid ? __ldg(p.rowptr + v + 1) : 0;
        const uint32_t pv = (p.prio && valid) ? __ldg(p.prio + v) : 0u;
        bool mine = false;
        const int rows = (int)min(R, (int64_t)nd - t0);
        for (int j = 0; j < rows; ++j) {
            const int32_t vj = __shfl_sync(kFull, v, j), bj = __shfl_sync(kFull, b, j), ej = __shfl_sync(kFull, e, j);
            const uint32_t pvj = __shfl_sync(kFull, pv, j);
            bool conflict = false;
            for (int32_t c = bj; c < ej && !conflict; c += 128) {
                int32_t w[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int32_t x = c + 32 * u + (int32_t)lane;
                    w[u] = x < ej ? ld_adj(p.colidx + x, pol_adj) : -1;
                }
                bool h = false;
#pragma unroll
                for (int u = 0; u < 4; ++u) h |= w[u] >= 0 && precedes(p.prio, w[u], vj, pvj);
                conflict = __any_sync(kFull, h);
            }
            if ((int)lane == j) mine = conflict;
        }
        if (valid) {
            pass1_write(p, v, mine, maxc);
            if (mine) vol += (unsigned)(e - b);
        }
        warp_append_hubs(nl, valid && mine, make_int4(v, b, e - b, e - b));
    }
    fold_max_color(p.st, maxc);
    fold_volume(p.st, p.round_vol, p.round_cap, 2, vol);
}

// ------------------------------------------------- fused pass, k >= 2

template <typename T>
struct PassIO {
    const T* Xc;            // C_k (flagged once settled)
    T* Xcw;                 // the same array, for setting the settled flag
    T* Xn;                  // receives C_{k+1}
    int k;                  // the round whose Phase 2 this pass runs
    const int32_t* rin;     // active lists read this round (colidx in round 2)
    int32_t* rout;          // active lists written for the next round
    bool first;             // round 2: no static masks yet
    const int4* L2; const int4* L4; const int4* L8; const int4* L16;
    const int4* S; const int4* M; const int4* H; const int32_t* Hc; const int32_t* O;
    NextLists next;
    uint64_t pol_row, pol_col;
};

template <typename T>
__device__ __forceinline__ PassIO<T> pass_io(const Params<T>& p, int k) {
    PassIO<T> io;
    const bool odd = (k & 1) != 0;
    io.Xc = odd ? p.X1 : p.X0;
    io.Xcw = odd ? p.X1 : p.X0;
    io.Xn = odd ? p.X0 : p.X1;
    io.first = k == 2;
    io.k = k;
    io.rin = k == 2 ? p.colidx : (odd ? p.act1 : p.act0);
    io.rout = odd ? p.act0 : p.act1;
    io.L2 = odd ? p.L2B : p.L2A;
    io.L4 = odd ? p.L4B : p.L4A;
    io.L8 = odd ? p.L8B : p.L8A;
    io.L16 = odd ? p.L16B : p.L16A;
    io.S = odd ? p.SB : p.SA;
    io.M = odd ? p.MB : p.MA;
    io.H = odd ? p.HB : p.HA;
    io.Hc = odd ? p.HcB : p.HcA;
    io.O = odd ? p.OB : p.OA;
    io.next.L2 = odd ? p.L2A : p.L2B;
    io.next.L4 = odd ? p.L4A : p.L4B;
    io.next.L8 = odd ? p.L8A : p.L8B;
    io.next.L16 = odd ? p.L16A : p.L16B;
    io.next.S = odd ? p.SA : p.SB;
    io.next.M = odd ? p.MA : p.MB;
    io.next.H = odd ? p.HA : p.HB;
    io.next.Hc = odd ? p.HcA : p.HcB;
    io.next.O = odd ? p.OA : p.OB;
    io.next.cnt = &p.st->rc[(k + 1) % 3];
    io.next.s_max = p.s_max;
    io.next.m_max = p.m_max;
    io.pol_row = policy_evict_first();
    io.pol_col = policy_evict_last();
    return io;
}

// v settles with color cv: flag it in both buffers, publish it.
template <typename T>
__device__ __forceinline__ void settle(const Params<T>& p, const PassIO<T>& io, int32_t v, uint32_t cv) {
    const T word = (T)(cv | Word<T>::kFlag);
    io.Xn[v] = word;
    io.Xcw[v] = word;
    p.colors_out[v] = (int32_t)cv;
    if (p.settle_round) p.settle_round[v] = io.k;
}

// v takes color c in round k+1.
template <typename T>
__device__ __forceinline__ void recolor(const Params<T>& p, const PassIO<T>& io, int32_t v, uint32_t c) {
    if (c >= p.color_limit) {
        atomicExch(&p.st->status, kStatusColorOverflow);
        io.next.cnt->overflow = 1u;
    }
    io.Xn[v] = (T)(c & (Word<T>::kFlag - 1u));
}

// What a warp needs to start a task.  Loaded one task ahead.
struct TaskHead {
    int4 e;       // worklist entry; x < 0 marks an empty slot
    int32_t pos;  // H chunk: worklist position of its vertex
    int32_t lo;   // H chunk: first entry of the chunk
};

// The entries of one round.
struct RoundSizes {
    unsigned n2, n4, n8, n16, nS, nM, nHC;  // L2, L4, L8, L16, S, M entries; H chunks
    unsigned overflow;
};
__device__ __forceinline__ RoundSizes round_sizes_of(const RoundCounts& c, unsigned* total) {
    RoundSizes r;
    const unsigned long long hc = __ldcg(&c.hc), tiny = __ldcg(&c.tiny), mid = __ldcg(&c.mid);
    r.n2 = low_count(tiny);
    r.n4 = high_count(tiny);
    r.overflow = __ldcg(&c.overflow);
    r.n8 = low_count(mid);
    r.n16 = high_count(mid);
    r.nS = __ldcg(&c.s);
    r.nM = __ldcg(&c.m);
    r.nHC = hub_chunks(hc);
    *total = r.n2 + r.n4 + r.n8 + r.n16 + r.nS + r.nM + hub_count(hc);
    return r;
}

// Its tasks, in the order they are dealt out: H chunks, M, L16, L8, S, L4, L2.
struct TaskSplit {
    unsigned mpt, spt;              // M and S entries per task
    unsigned s16, s8, s4, s2;       // steps per task of L16, L8, L4 and L2
    unsigned e0, e1, e2, e3, e4, e5;  // ends of the H, M, L16, L8, S and L4 tasks
    unsigned total;
    unsigned nstat;                 // tasks a warp takes without a claim
};

// Entry of step j < steps of a row task: lane j of every group of L lanes
// holds the entry that the group takes in step j.
template <int L>
__device__ __forceinline__ unsigned step_entry(unsigned t, unsigned steps, unsigned* j) {
    *j = lane_id() % L;
    return (t * steps + *j) * (32 / L) + lane_id() / L;
}

template <typename T>
__device__ __forceinline__ TaskHead load_head(const PassIO<T>& io, unsigned t, const RoundSizes& r,
                                              const TaskSplit& q) {
    TaskHead h;
    h.pos = 0;
    h.lo = 0;
    if (t < q.e0) {
        h.pos = __ldcg(io.O + t);
        h.e = __ldcg(io.H + h.pos);
        h.lo = h.e.y + ((int32_t)t - __ldcg(io.Hc + h.pos)) * kChunk;
        return h;
    }
    const int4* list;
    unsigned i, n, j = lane_id(), most;
    if (t < q.e1) {
        list = io.M; n = r.nM; most = q.mpt; i = (t - q.e0) * q.mpt + j;
    } else if (t < q.e2) {
        list = io.L16; n = r.n16; most = q.s16; i = step_entry<16>(t - q.e1, q.s16, &j);
    } else if (t < q.e3) {
        list = io.L8; n = r.n8; most = q.s8; i = step_entry<8>(t - q.e2, q.s8, &j);
    } else if (t < q.e4) {
        list = io.S; n = r.nS; most = q.spt; i = (t - q.e3) * q.spt + j;
    } else if (t < q.e5) {
        list = io.L4; n = r.n4; most = q.s4; i = step_entry<4>(t - q.e4, q.s4, &j);
    } else {
        list = io.L2; n = r.n2; most = q.s2; i = step_entry<2>(t - q.e5, q.s2, &j);
    }
    h.e = j < most && i < n ? __ldcg(list + i) : make_int4(-1, 0, 0, 0);
    return h;
}

// Shared memory of one warp for a flat task.
// The color windows are stored word-major ([word q][lane]), so the 32 lanes
// touching word q of their own vertex's window hit 32 different banks.
struct FlatSmem {
    uint32_t stat[8 * 32];  // per entry vertex: static mask (+ colors settled this round)
    uint32_t dyn[8 * 32];   // per entry vertex: colors of unsettled neighbours this round
    uint32_t conf;          // per entry vertex: conflict flag
    uint32_t lane_of[32];   // lane of the i-th non-empty row
    int32_t vid[32];        // vertex of each lane
};

// Ask L1 for the line holding a (list entries read soon by this warp).
__device__ __forceinline__ void prefetch_l1(const void* a) {
    asm volatile("prefetch.global.L1 [%0];" :: "l"(a));
}

// Stores of the next round's active lists and static masks: read once, in
// the next round, so evicted first.
__device__ __forceinline__ void st_stream(int32_t* a, int32_t x, uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.s32 [%0], %1, %2;" :: "l"(a), "r"(x), "l"(pol) : "memory");
}

// The state of an L2 or L4 entry in its last two words.  With a priority array
// the rows have at most kKeyedBits = 21 entries, so that the live bits, the
// precedence bits and the mask of the colors 1..22 fill the 64 bits.
template <bool P>
struct TinyState {
    uint32_t live, prec, stat;
    __device__ __forceinline__ static TinyState of(int4 e) {
        const uint32_t z = (uint32_t)e.z, w = (uint32_t)e.w;
        if constexpr (!P) return {z, 0u, w};
        return {z & ((1u << kKeyedBits) - 1u), (z >> kKeyedBits) | ((w & 0x3ffu) << 11), w >> 10};
    }
    __device__ __forceinline__ int4 entry(int32_t v, int32_t b) const {
        if constexpr (!P) return make_int4(v, b, (int32_t)live, (int32_t)stat);
        return make_int4(v, b, (int32_t)(live | prec << kKeyedBits), (int32_t)(prec >> 11 | stat << 10));
    }
};

// L2 and L4 bins (L = 2, 4): vertices of degree <= 8 L - 7 <= 25 (and s_max),
// whose first fit is at most 26, so one 32-bit word holds every color that matters to them and one more says
// which entries of the row are still live (the neighbour had not settled when
// last read).  Both travel in the worklist entry {v, row start, live, static
// mask}, with a priority array beside one bit per entry for "precedes v"
// (TinyState); the row itself is read from colidx in every round and no list
// is written.
//
// L lanes share a vertex: each takes a 32-byte chunk of the row (one load for
// eight entries; a row of 8 L - 7 spans at most L), gathers the colors of the live entries, and ORs
// what it finds in registers; the lanes of a vertex combine with shuffles.
// Lane j of a group keeps the vertex of step j, so a task of up to 32
// vertices appends its survivors with one atomic.
//
// Two lanes for rows of up to 9 (a mesh's, say) fill twice the lanes of four:
// 5-point mesh of 4,000,003 vertices 0.55 -> 0.46 ms.
//
// Bound: the random L2 sector of each live entry's color (207 G entries/s on
// rows of 16; a probe that only gathers reaches 208).  The flat walk below,
// which these rows took before, ran at 133 G entries/s: 157 instructions per
// 32 entries against about 40 here, and an L1 data pipe 72 % busy, two fifths
// of it with shared-memory atomics.  R-MAT-ER of 2^22 vertices: 2.36 ms a call
// before, 1.70 after.
template <typename T, bool P, int L>  // P: a priority array is given
__device__ __forceinline__ void tiny_task(const Params<T>& p, const PassIO<T>& io, int4 en, unsigned steps, int& maxc,
                                          unsigned& vol) {
    const unsigned lane = lane_id();
    const unsigned j = lane % L;
    const uint32_t mis = (uint32_t)((uintptr_t)p.colidx >> 2) & 7u;  // entries from a 32-byte boundary to colidx
    const bool valid = en.x >= 0;
    const int32_t my_v = valid ? en.x : 0;
    const TinyState<P> my = TinyState<P>::of(valid ? en : make_int4(0, 0, 0, 0));
    const uint32_t my_live = my.live;
    const uint32_t my_cv = valid ? word_color(ld_color(io.Xc + my_v, io.pol_col)) : 0u;
    // which entries precede v (bit i: entry i), worked out in round 2; there: v's key
    const uint32_t my_prec = P && io.first ? (valid ? __ldg(p.prio + my_v) : 0u) : my.prec;
    uint32_t my_all = 0u, my_stat = 0u, my_dead = 0u, my_new_prec = 0u;
    bool my_conflict = false;
#pragma unroll 1
    for (unsigned s = 0; s < steps; ++s) {
        const int src = (int)((lane & ~(unsigned)(L - 1)) | s);
        const int32_t v = __shfl_sync(kFull, my_v, src);
        const int32_t b = __shfl_sync(kFull, en.y, src);
        const uint32_t live = __shfl_sync(kFull, my_live, src);
        uint32_t all = 0u, stat = 0u, dead = 0u, nprec = 0u;
        bool conflict = false;
        // this lane's chunk: entries off .. off + 7 of the row (the first chunk may
        // start before the row); bits: the live ones
        const int32_t off = 8 * (int32_t)j - (int32_t)(((uint32_t)b + mis) & 7u);
        const uint32_t bits = (off >= 0 ? live >> off : live << -off) & 0xffu;
        const uint32_t cv = __shfl_sync(kFull, my_cv, src);
        const uint32_t prec = P ? __shfl_sync(kFull, my_prec, src) : 0u;
        if (bits) {
            int32_t w[8];
            load_chunk(p.colidx, p.nnz, b + off, io.pol_row, w);
            T c[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) c[u] = (bits >> u) & 1u ? ld_color(io.Xc + w[u], io.pol_col) : (T)0;
            uint32_t gone = 0u, pre8 = 0u;
            if constexpr (P) {
                if (!io.first) {
                    pre8 = off >= 0 ? prec >> off : prec << -off;
                } else {
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        if (((bits >> u) & 1u) && (word_color(c[u]) == cv || !word_settled(c[u])) &&
                            precedes(p.prio, w[u], v, prec))
                            pre8 |= 1u << u;
                    nprec = off >= 0 ? pre8 << off : pre8 >> -off;
                }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const uint32_t col = word_color(c[u]);         // 0 where the entry is not live
                const uint32_t bit = shl_clamp(1u, col - 1u);  // 0 for col 0 and col > 32
                all |= bit;
                if (word_settled(c[u])) {
                    stat |= bit;
                    gone |= 1u << u;
                }
                if (col == cv && (P ? (pre8 >> u) & 1u : w[u] < v)) conflict = true;
            }
            dead = off >= 0 ? gone << off : gone >> -off;
        }
        const unsigned cb = __ballot_sync(kFull, conflict);
#pragma unroll
        for (int o = 1; o < L; o <<= 1) {
            all |= __shfl_xor_sync(kFull, all, o);
            stat |= __shfl_xor_sync(kFull, stat, o);
            dead |= __shfl_xor_sync(kFull, dead, o);
            if (P && io.first) nprec |= __shfl_xor_sync(kFull, nprec, o);
        }
        if (j == s) {
            my_all = all;
            my_stat = stat;
            my_dead = dead;
            my_new_prec = nprec;
            my_conflict = ((cb >> (lane - j)) & ((1u << L) - 1u)) != 0u;
        }
    }
    const bool go = valid && my_conflict;
    TinyState<P> now;
    now.live = my_live & ~my_dead;
    now.prec = P && io.first ? my_new_prec : my.prec;
    now.stat = my.stat | (P ? my_stat & ((1u << (kKeyedBits + 1)) - 1u) : my_stat);  // (first fit is at most 22)
    if (go) {
        recolor(p, io, my_v, (uint32_t)__ffs(~(now.stat | my_all)));
        vol += (unsigned)__popc(now.live);
    } else if (valid) {
        settle(p, io, my_v, my_cv);
        maxc = max(maxc, (int)my_cv);
    }
    warp_append_pair<(L == 2 ? 0 : 32)>(go, now.entry(my_v, en.y),
                                        L == 2 ? io.next.L2 : io.next.L4, &io.next.cnt->tiny);
}

// L8 and L16 bins (L = 8, 16): longer rows of degree d <= 8 L - 7, read
// like the short rows: L lanes share a vertex, one 32-byte chunk of colidx each, 32 / L
// vertices side by side, no list written.  Their first fit is at most
// 8 L - 6, so W = L / 4 words hold the colors that matter.  The static mask
// (words 0..W-1) and one byte of live entries per chunk (after it) share the
// vertex's 32 bytes of p.stat; with a priority array, one byte more per chunk
// says which entries precede v (L8: after the live bytes; L16: in p.act0's part
// of the row, which no list of this vertex uses).
//
// Bound: as for the short rows, one random L2 sector per live entry.  A warp per
// vertex (the M bin, which these rows took before) leaves most of its lanes
// without an entry on a list of 33..64 and repeats its per-vertex work 32
// wide: 98 G entries/s on rows of 48 and 158 on rows of 96, against 214 and
// 227 here; on rows of 192 the two are level (200), so longer rows stay there.
// R-MAT-B of 2^24 vertices: 24.34 -> 22.40 ms a call, learned R-MAT-G of 2^23:
// 17.15 -> 14.07 ms.
template <typename T, bool P, int L>  // P: a priority array is given
__device__ __forceinline__ void mid_task(const Params<T>& p, const PassIO<T>& io, int4 en, unsigned steps, int& maxc,
                                         unsigned& vol) {
    constexpr int W = L / 4;
    const unsigned lane = lane_id();
    const unsigned j = lane % L;
    const uint32_t mis = (uint32_t)((uintptr_t)p.colidx >> 2) & 7u;
    const bool first = io.first;
    const bool valid = en.x >= 0;
    const int32_t my_v = valid ? en.x : 0;
    const int32_t my_d = valid ? en.z : 0;  // 0: nothing to read
    bool my_conflict = false;
    uint32_t my_color = 0u, my_cv = 0u;
#pragma unroll 1
    for (unsigned s = 0; s < steps; ++s) {
        const int src = (int)((lane & ~(unsigned)(L - 1)) | s);
        const int32_t v = __shfl_sync(kFull, my_v, src);
        const int32_t b = __shfl_sync(kFull, en.y, src);
        const int32_t d = __shfl_sync(kFull, my_d, src);
        // every lane reads v's color itself, so that the row's load does not wait for it
        // (one line either way)
        const uint32_t cv = d ? word_color(ld_color(io.Xc + v, io.pol_col)) : 0u;
        const uint32_t key = P && first && d ? __ldg(p.prio + v) : 0u;
        // this lane's chunk: entries off .. off + 7 of the row
        const int32_t off = 8 * (int32_t)j - (int32_t)(((uint32_t)b + mis) & 7u);
        uint32_t* const st = p.stat + (size_t)v * 8;
        uint8_t* const live_at = reinterpret_cast<uint8_t*>(st + W) + j;
        uint8_t* const prec_at = (L == 8 ? reinterpret_cast<uint8_t*>(st + 2 * W) : reinterpret_cast<uint8_t*>(p.act0 + b)) + j;
        uint32_t live, old = 0u, prec = 0u;
        if (first) {
            live = low_bits(max(0, min(8, d - off))) & (off < 0 ? 0xffu << -off : 0xffu);
        } else {
            live = d ? (uint32_t)__ldcg(live_at) : 0u;
            if (d && j < W) old = __ldcg(st + j);
            if (P && d) prec = (uint32_t)__ldcg(prec_at);
        }
        uint32_t all[W], stat[W], gone = 0u;
#pragma unroll
        for (int q = 0; q < W; ++q) {
            all[q] = 0u;
            stat[q] = (int)j == q ? old : 0u;
        }
        bool conflict = false;
        if (live) {
            int32_t w[8];
            load_chunk(p.colidx, p.nnz, b + off, io.pol_row, w);
            T c[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) c[u] = (live >> u) & 1u ? ld_color(io.Xc + w[u], io.pol_col) : (T)0;
            if (P && first) {
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (((live >> u) & 1u) && (word_color(c[u]) == cv || !word_settled(c[u])) &&
                        precedes(p.prio, w[u], v, key))
                        prec |= 1u << u;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const uint32_t col = word_color(c[u]);  // 0 where the entry is not live
#pragma unroll
                for (int q = 0; q < W; ++q) all[q] |= shl_clamp(1u, col - 1u - 32u * q);
                if (word_settled(c[u])) {
                    gone |= 1u << u;
#pragma unroll
                    for (int q = 0; q < W; ++q) stat[q] |= shl_clamp(1u, col - 1u - 32u * q);
                }
                if (col == cv && (P ? (prec >> u) & 1u : w[u] < v)) conflict = true;
            }
        }
        const unsigned cb = __ballot_sync(kFull, conflict);
        const bool conf = ((cb >> (lane - j)) & low_bits(L)) != 0u;
#pragma unroll
        for (int o = 1; o < L; o <<= 1)
#pragma unroll
            for (int q = 0; q < W; ++q) {
                all[q] |= __shfl_xor_sync(kFull, all[q], o);
                stat[q] |= __shfl_xor_sync(kFull, stat[q], o);
            }
        uint32_t color = 0u, mine = 0u;  // v's next color; this lane's word of the static mask
#pragma unroll
        for (int q = W - 1; q >= 0; --q) {
            const uint32_t taken = all[q] | stat[q];
            if (taken != 0xffffffffu) color = 32u * q + (uint32_t)__ffs(~taken);
            if ((int)j == q) mine = stat[q];
        }
        if (conf) {
            const uint32_t now = live & ~gone;
            if (j < W && (first || mine != old)) st[j] = mine;
            if (first || gone) *live_at = (uint8_t)now;
            if (P && first) *prec_at = (uint8_t)prec;
            vol += (unsigned)__popc(now);
        }
        if (j == s) {
            my_cv = cv;
            my_conflict = conf;
            my_color = color;
        }
    }
    const bool go = valid && my_conflict;
    if (go) {
        recolor(p, io, my_v, my_color);
    } else if (valid) {
        settle(p, io, my_v, my_cv);
        maxc = max(maxc, (int)my_cv);
    }
    warp_append_pair<(L == 8 ? 0 : 32)>(go, en, L == 8 ? io.next.L8 : io.next.L16, &io.next.cnt->mid);
}

// S bin: up to 32 worklist entries per task, one per lane.  Their
// active lists are walked as one flat range in batches of 32 entries (lane
// l of batch u takes flat entry F0 + 32u + l), so every lane has an entry in
// every batch whatever the lengths are.  The row owning an entry is found
// from the batch's row starts: a row that starts inside the batch sets the
// bit of its first lane (one OR-reduction over the warp), and an entry's
// row is the last one started at or before it, counted among the non-empty
// rows (a 32-entry table maps that count to the row's lane).  Each entry ORs its neighbour's color into
// its vertex's window in shared memory, flags a conflict, and, if the
// neighbour has not settled, is copied to the next round's list at the
// vertex's running write position.  Afterwards each lane decides its own
// vertex.  Round 2 has no S entries: pass 1 gives rows of up to s_max to the L2,
// L4 and L8 bins, so every vertex here has a static mask, and with keys every
// entry carries its precedence bit.
template <typename T, bool P>  // P: a priority array is given
__device__ __forceinline__ void flat_task(const Params<T>& p, const PassIO<T>& io, int4 en,
                                          FlatSmem& sm, int& maxc, unsigned& vol) {
    const unsigned lane = lane_id();
    const bool valid = en.x >= 0;
    const int32_t v = valid ? en.x : 0;
    const int32_t b = en.y;
    const int32_t len = valid ? en.z : 0;
    const uint32_t cv = valid ? word_color(ld_color(io.Xc + v, io.pol_col)) : 0u;
    // static mask of v
    if (valid) {
        const uint4* src = reinterpret_cast<const uint4*>(p.stat + (size_t)v * 8);
        const uint4 a = __ldcg(src), c = __ldcg(src + 1);
        sm.stat[0 * 32 + lane] = a.x; sm.stat[1 * 32 + lane] = a.y;
        sm.stat[2 * 32 + lane] = a.z; sm.stat[3 * 32 + lane] = a.w;
        sm.stat[4 * 32 + lane] = c.x; sm.stat[5 * 32 + lane] = c.y;
        sm.stat[6 * 32 + lane] = c.z; sm.stat[7 * 32 + lane] = c.w;
    } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) sm.stat[q * 32 + lane] = 0u;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) sm.dyn[q * 32 + lane] = 0u;
    if (lane == 0) sm.conf = 0u;
    int32_t incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t x = __shfl_up_sync(kFull, incl, o);
        if ((int)lane >= o) incl += x;
    }
    const int32_t off = incl - len;
    const int32_t D = __shfl_sync(kFull, incl, 31);
    const unsigned nz = __ballot_sync(kFull, len > 0);  // rows that own entries
    if (len > 0) sm.lane_of[__popc(nz & ((1u << lane) - 1u))] = lane;
    sm.vid[lane] = v;
    int32_t kept = 0;  // entries of this lane's vertex written for the next round
    __syncwarp();
    const int32_t b_off = b - off;  // row start minus flat offset: entry f of this row is at b_off + f
    for (int32_t F0 = 0; F0 < D; F0 += 32 * kFlatBatches) {
        int32_t w[kFlatBatches], own[kFlatBatches], seglo[kFlatBatches];
#pragma unroll
        for (int u = 0; u < kFlatBatches; ++u) {
            const int32_t base = F0 + 32 * u;
            const int32_t f = base + (int32_t)lane;
            // rows started before this batch, and the starts inside it
            const int32_t rel = off - base;
            const unsigned before = __popc(__ballot_sync(kFull, len > 0 && rel < 0));
            const unsigned starts = __reduce_or_sync(kFull, (len > 0 && rel >= 0 && rel < 32) ? (1u << rel) : 0u);
            const unsigned upto = starts & (0xffffffffu >> (31 - lane));
            const unsigned rank = before + __popc(upto);
            const int o = (f < D && rank > 0) ? (int)sm.lane_of[rank - 1] : 0;
            own[u] = o;
            // first lane of my owner's entries in this batch: the last row start at or
            // before this lane, or 0 if the row began in an earlier batch
            seglo[u] = upto ? 31 - __clz(upto) : 0;
            const int32_t rb = __shfl_sync(kFull, b_off, o);
            w[u] = f < D ? ld_row(io.rin + rb + f, io.pol_row) : 0;
        }
        T c[kFlatBatches];
#pragma unroll
        for (int u = 0; u < kFlatBatches; ++u) {
            const int32_t f = F0 + 32 * u + (int32_t)lane;
            c[u] = f < D ? ld_color(io.Xc + (P ? entry_id(w[u]) : w[u]), io.pol_col) : (T)0;
        }
#pragma unroll
        for (int u = 0; u < kFlatBatches; ++u) {
            const int32_t base = F0 + 32 * u;
            const int32_t f = base + (int32_t)lane;
            const int o = own[u];
            const uint32_t ocv = __shfl_sync(kFull, cv, o);
            const int32_t wbase = __shfl_sync(kFull, b + kept, o);  // next free slot of the owner's list
            const bool in = f < D;
            const uint32_t col = word_color(c[u]);
            const bool settled = in && word_settled(c[u]);
            // (with keys, an entry's bit says that it precedes its owner)
            if (in && col == ocv && (P ? w[u] < 0 : w[u] < sm.vid[o])) atomicOr(&sm.conf, 1u << o);
            {
                const unsigned idx = col - 1u;
                if (in && idx < 256u)
                    atomicOr(settled ? &sm.stat[(idx >> 5) * 32 + o] : &sm.dyn[(idx >> 5) * 32 + o],
                             1u << (idx & 31u));
            }
            // survivors: copy to the next round's list, in order within each vertex
            const bool keep = in && !settled;
            const unsigned kb = __ballot_sync(kFull, keep);
            const unsigned below = kb & ((1u << lane) - 1u) & ~((1u << seglo[u]) - 1u);
            if (keep)
                st_stream(io.rout + wbase + __popc(below), w[u], io.pol_row);
            // my vertex's lanes in this batch: [lo, hi)
            const int32_t lo = max(0, min(32, off - base));
            const int32_t hi = max(0, min(32, off + len - base));
            if (hi > lo) {
                const unsigned bits = hi - lo == 32 ? kFull : ((1u << (hi - lo)) - 1u);
                kept += __popc((kb >> lo) & bits);
            }
        }
    }
    __syncwarp();
    const bool conflict = valid && ((sm.conf >> lane) & 1u);
    uint32_t color = 0;
    bool rescan = false;
    if (conflict) {
        int ff = -1;
#pragma unroll
        for (int q = 7; q >= 0; --q) {
            const uint32_t word = sm.stat[q * 32 + lane] | sm.dyn[q * 32 + lane];
            if (word != 0xffffffffu) ff = q * 32 + __ffs(~word) - 1;
        }
        if (ff >= 0) color = (uint32_t)ff + 1u;
        else rescan = true;
    }
    unsigned need = __ballot_sync(kFull, rescan);
    while (need) {
        const int j = __ffs(need) - 1;
        need &= need - 1;
        const uint32_t cj = rescan_first_fit(p.rowptr, p.colidx, io.Xc, __shfl_sync(kFull, v, j));
        if ((int)lane == j) color = cj;
    }
    if (valid) {
        if (conflict) {
            recolor(p, io, v, color);
            vol += (unsigned)kept;
            uint4* dst = reinterpret_cast<uint4*>(p.stat + (size_t)v * 8);
            dst[0] = make_uint4(sm.stat[0 * 32 + lane], sm.stat[1 * 32 + lane],
                                sm.stat[2 * 32 + lane], sm.stat[3 * 32 + lane]);
            dst[1] = make_uint4(sm.stat[4 * 32 + lane], sm.stat[5 * 32 + lane],
                                sm.stat[6 * 32 + lane], sm.stat[7 * 32 + lane]);
        } else {
            settle(p, io, v, cv);
            maxc = max(maxc, (int)cv);
        }
    }
    // next round: same row start, `kept` active entries; the bin may shrink
    const int4 ne = make_int4(v, b, kept, en.w);
    const int nb = bin_of(kept, p.s_max, p.m_max);
    warp_append(conflict && nb == kBinS, ne, io.next.S, &io.next.cnt->s);
    warp_append(conflict && nb == kBinM, ne, io.next.M, &io.next.cnt->m);
    __syncwarp();
}

// M bin: up to kMedPerTask worklist entries per task (lane i holds entry i), taken
// one vertex at a time by the whole warp: lane l reads entries l, l + 32, ...
// of the vertex's active list, four batches of 32 in flight.  Colors 1..64
// collect in per-lane registers (all neighbours, and those found settled)
// and are OR-reduced once per vertex; colors 65..256 go to the warp's shared
// windows, where no two vertices meet.  So the lanes never contend on one
// shared word, which the flat walk does when most of a batch belongs to one
// long list.  The decisions stay in the lane of their entry, and the task
// appends its conflicting vertices to the next round with one atomic per
// bin.  Round 2 with keys (F: keys are compared and kept as a bit of the entry)
// is an instance of its own here and in hub_chunk; the later rounds then run
// without its branches, which matters where most entries stand in lists: with
// keys by features and R-MAT-B at 4M vertices 10.63 ms in one instance, 10.35 ms
// in two; short-row graphs (G(1M, 8M), R-MAT-G at 8M) are unchanged.
template <typename T, bool P, bool F>  // P: a priority array is given; F: and this is round 2
__device__ __forceinline__ void vertex_task(const Params<T>& p, const PassIO<T>& io, int4 en,
                                            FlatSmem& sm, int& maxc, unsigned& vol) {
    constexpr int kB = 4;  // batches in flight
    const unsigned lane = lane_id();
    const bool first = io.first;
    bool my_conflict = false;
    int32_t my_kept = 0;
    unsigned todo = __ballot_sync(kFull, en.x >= 0);
    while (todo) {
        const int j = __ffs(todo) - 1;
        todo &= todo - 1;
        const int32_t v = __shfl_sync(kFull, en.x, j);
        const int32_t b = __shfl_sync(kFull, en.y, j);
        const int32_t len = __shfl_sync(kFull, en.z, j);
        // the next vertex's list comes into L1 while this one is read (lanes 0..8:
        // one 128-byte line each, the last one for the end of the list)
        if (todo) {
            const int jn = __ffs(todo) - 1;
            const int32_t bn = __shfl_sync(kFull, en.y, jn), ln = __shfl_sync(kFull, en.z, jn);
            if (lane < 8u && (int32_t)lane * 32 < ln) prefetch_l1(io.rin + bn + 32 * lane);
            else if (lane == 8u) prefetch_l1(io.rin + bn + ln - 1);
        }
        const uint32_t cv = word_color(ld_color(io.Xc + v, io.pol_col));
        const uint32_t pv = F ? __ldg(p.prio + v) : 0u;
        // v's static mask, word `lane` (read now, used after the list)
        const uint32_t old = (lane < 8u && !first) ? __ldcg(p.stat + (size_t)v * 8 + lane) : 0u;
        if (lane < 8u) { sm.dyn[lane] = 0u; sm.stat[lane] = 0u; }
        __syncwarp();
        uint32_t rd0 = 0u, rs0 = 0u, rd1 = 0u, rs1 = 0u;  // this lane's colors 1..64 (all, settled)
        bool conflict = false;
        int32_t kept = 0;
        for (int32_t base = 0; base < len; base += 32 * kB) {
            int32_t w[kB];
            T c[kB];
#pragma unroll
            for (int u = 0; u < kB; ++u) {
                const int32_t i = base + 32 * u + (int32_t)lane;
                w[u] = i < len ? ld_row(io.rin + b + i, io.pol_row) : 0;
            }
#pragma unroll
            for (int u = 0; u < kB; ++u) {
                const int32_t i = base + 32 * u + (int32_t)lane;
                c[u] = i < len ? ld_color(io.Xc + (P ? entry_id(w[u]) : w[u]), io.pol_col) : (T)0;
            }
#pragma unroll
            for (int u = 0; u < kB; ++u) {
                const int32_t i = base + 32 * u + (int32_t)lane;
                const bool in = i < len;
                const uint32_t col = word_color(c[u]);
                const bool settled = in && word_settled(c[u]);
                const int32_t wid = P ? entry_id(w[u]) : w[u];
                bool pre = false;
                if constexpr (!P) {
                    pre = in && col == cv && wid < v;
                } else if (in && (col == cv || (F && !settled))) {
                    pre = F ? precedes(p.prio, wid, v, pv) : w[u] < 0;
                    if (F) w[u] = (int32_t)((uint32_t)wid | (pre ? kPrecBit : 0u));  // the entry kept
                }
                if (in) {
                    if (col == cv && pre) conflict = true;
                    const unsigned idx = col - 1u;
                    const uint32_t bit = 1u << (idx & 31u);
                    if (idx < 32u) {
                        rd0 |= bit;
                        rs0 |= settled ? bit : 0u;
                    } else if (idx < 64u) {
                        rd1 |= bit;
                        rs1 |= settled ? bit : 0u;
                    } else if (idx < 256u) {
                        atomicOr(&sm.dyn[idx >> 5], bit);
                        if (settled) atomicOr(&sm.stat[idx >> 5], bit);
                    }
                }
                // survivors, in order, to the next round's list
                const unsigned kb = __ballot_sync(kFull, in && !settled);
                if (in && !settled)
                    st_stream(io.rout + b + kept + __popc(kb & ((1u << lane) - 1u)), w[u], io.pol_row);
                kept += __popc(kb);
            }
        }
        const bool conf = __any_sync(kFull, conflict);
        rd0 = __reduce_or_sync(kFull, rd0);
        rs0 = __reduce_or_sync(kFull, rs0);
        rd1 = __reduce_or_sync(kFull, rd1);
        rs1 = __reduce_or_sync(kFull, rs1);
        __syncwarp();
        const unsigned q7 = lane & 7u;
        uint32_t stat = 0u, all = 0u;
        if (lane < 8u) {
            stat = old | sm.stat[q7] | (q7 == 0u ? rs0 : (q7 == 1u ? rs1 : 0u));
            all = stat | sm.dyn[q7] | (q7 == 0u ? rd0 : (q7 == 1u ? rd1 : 0u));
        }
        __syncwarp();
        if (!conf) {
            if (lane == 0) settle(p, io, v, cv);
            maxc = max(maxc, (int)cv);
        } else {
            const int ff = window_first_clear(all);
            const uint32_t color = ff >= 0 ? (uint32_t)ff + 1u : rescan_first_fit(p.rowptr, p.colidx, io.Xc, v);
            if (lane < 8u) p.stat[(size_t)v * 8 + lane] = stat;
            if (lane == 0) {
                recolor(p, io, v, color);
                vol += (unsigned)kept;
            }
        }
        if ((int)lane == j) {
            my_conflict = conf;
            my_kept = kept;
        }
    }
    // next round: same row start, the kept entries; the bin may shrink (never grow)
    const int4 ne = make_int4(en.x, en.y, my_kept, en.w);
    const int nb = bin_of(my_kept, p.s_max, p.m_max);
    warp_append(my_conflict && nb == kBinS, ne, io.next.S, &io.next.cnt->s);
    warp_append(my_conflict && nb == kBinM, ne, io.next.M, &io.next.cnt->m);
    __syncwarp();
}

// H bin: one chunk of up to 1024 entries of the vertex at worklist position
// h.pos, read in sub-blocks of 256 (two halves of 4 entries per lane).  A
// vertex whose active list fits one chunk is decided by this warp at once;
// otherwise the chunks OR their results into the vertex's record, and the
// warp that completes the last chunk decides it and clears the record.
template <typename T, bool P, bool F>  // P: a priority array is given; F: and this is round 2
__device__ __forceinline__ void hub_chunk(const Params<T>& p, const PassIO<T>& io, TaskHead h,
                                          FlatSmem& sm, int& maxc, unsigned& vol) {
    constexpr int kHalf = kPerLane / 2;
    const unsigned lane = lane_id();
    const int32_t v = h.e.x, b = h.e.y, len = h.e.z;
    const int32_t e = b + len;
    const int32_t lo = h.lo, hi = min(e, lo + kChunk);
    const unsigned nch = (unsigned)(len + kChunk - 1) / kChunk;
    const bool single = nch == 1;
    const uint32_t cv = word_color(ld_color(io.Xc + v, io.pol_col));
    const uint32_t pv = F ? __ldg(p.prio + v) : 0u;
    // a vertex decided by this warp: its static mask word `lane`, read now
    const uint32_t old_single = (single && lane < 8u && !io.first) ? __ldcg(p.stat + (size_t)v * 8 + lane) : 0u;
    bool conflict = false;
    // this chunk's color windows: all colors in sm.dyn[0..8), settled ones in sm.stat[0..8)
    if (lane < 8u) { sm.dyn[lane] = 0u; sm.stat[lane] = 0u; }
    __syncwarp();
    HubRecord* rec = p.hubs + h.pos;
    unsigned local = 0;  // survivors written so far (single-chunk vertex)
    uint32_t rd0 = 0u, rs0 = 0u, rd1 = 0u, rs1 = 0u;  // this lane's colors 1..64 (all, settled)
    for (int32_t sb = lo; sb < hi; sb += kHubSub) {
        // the next sub-block (eight 128-byte lines) comes into L1 meanwhile
        if (lane < 8u && sb + kHubSub + 32 * (int32_t)lane < hi) prefetch_l1(io.rin + sb + kHubSub + 32 * lane);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            int32_t w[kHalf];
            T c[kHalf];
            unsigned keepbits[kHalf];
#pragma unroll
            for (int u = 0; u < kHalf; ++u) {
                const int32_t j = sb + (int32_t)lane + 32 * (half * kHalf + u);
                w[u] = j < hi ? ld_row(io.rin + j, io.pol_row) : 0;
            }
#pragma unroll
            for (int u = 0; u < kHalf; ++u) {
                const int32_t j = sb + (int32_t)lane + 32 * (half * kHalf + u);
                c[u] = j < hi ? ld_color(io.Xc + (P ? entry_id(w[u]) : w[u]), io.pol_col) : (T)0;
            }
            unsigned nkeep = 0;
#pragma unroll
            for (int u = 0; u < kHalf; ++u) {
                const int32_t j = sb + (int32_t)lane + 32 * (half * kHalf + u);
                const bool in = j < hi;
                const uint32_t col = word_color(c[u]);
                const bool settled = in && word_settled(c[u]);
                const int32_t wid = P ? entry_id(w[u]) : w[u];
                bool pre = false;
                if constexpr (!P) {
                    pre = in && col == cv && wid < v;
                } else if (in && (col == cv || (F && !settled))) {
                    pre = F ? precedes(p.prio, wid, v, pv) : w[u] < 0;
                    if (F) w[u] = (int32_t)((uint32_t)wid | (pre ? kPrecBit : 0u));  // the entry kept
                }
                if (in) {
                    if (col == cv && pre) conflict = true;
                    const unsigned idx = col - 1u;
                    // colors 1..64 gather in registers (one warp reduction per chunk); the
                    // rest go to the shared windows, where every lane of the warp would
                    // otherwise hit the same few words
                    const uint32_t bit = 1u << (idx & 31u);
                    if (idx < 32u) {
                        rd0 |= bit;
                        rs0 |= settled ? bit : 0u;
                    } else if (idx < 64u) {
                        rd1 |= bit;
                        rs1 |= settled ? bit : 0u;
                    } else if (idx < 256u) {
                        atomicOr(&sm.dyn[idx >> 5], bit);
                        if (settled) atomicOr(&sm.stat[idx >> 5], bit);
                    }
                }
                keepbits[u] = __ballot_sync(kFull, in && !settled);
                nkeep += __popc(keepbits[u]);
            }
            // survivors go to [b + slot, b + slot + nkeep) of the next round's list
            unsigned slot = local;
            if (!single) {
                if (lane == 0 && nkeep) slot = atomicAdd(&rec->kept, nkeep);
                slot = __shfl_sync(kFull, slot, 0);
            }
            local += nkeep;
#pragma unroll
            for (int u = 0; u < kHalf; ++u) {
                if ((keepbits[u] >> lane) & 1u)
                    st_stream(io.rout + b + slot + __popc(keepbits[u] & ((1u << lane) - 1u)), w[u], io.pol_row);
                slot += __popc(keepbits[u]);
            }
        }
    }
    const bool any_conflict = __any_sync(kFull, conflict);
    __syncwarp();
    rd0 = __reduce_or_sync(kFull, rd0);
    rs0 = __reduce_or_sync(kFull, rs0);
    rd1 = __reduce_or_sync(kFull, rd1);
    rs1 = __reduce_or_sync(kFull, rs1);
    const unsigned q7 = lane & 7u;
    const uint32_t word = sm.dyn[q7] | (q7 == 0u ? rd0 : (q7 == 1u ? rd1 : 0u));
    const uint32_t sword = sm.stat[q7] | (q7 == 0u ? rs0 : (q7 == 1u ? rs1 : 0u));
    __syncwarp();
    bool conf;
    int32_t kept;
    uint32_t all = 0, stat = 0;
    if (single) {
        conf = any_conflict;
        kept = (int32_t)local;
        if (lane < 8u) {
            stat = old_single | sword;
            all = stat | word;
        }
    } else {
        if (lane < 8u && word) atomicOr(&rec->mask[lane], word);
        if (lane < 8u && sword) atomicOr(&rec->stat[lane], sword);
        if (lane == 0 && any_conflict) atomicOr(&rec->conflict, 1u);
        __threadfence();
        unsigned done = 0;
        if (lane == 0) done = atomicAdd(&rec->done, 1u);
        done = __shfl_sync(kFull, done, 0);
        if (done != nch - 1) return;
        // last chunk of v: decide
        __threadfence();
        conf = __ldcg(&rec->conflict) != 0u;
        kept = (int32_t)__ldcg(&rec->kept);
        if (lane < 8u) {
            const uint32_t old = io.first ? 0u : __ldcg(p.stat + (size_t)v * 8 + lane);
            stat = old | __ldcg(&rec->stat[lane]);
            all = stat | __ldcg(&rec->mask[lane]);
        }
        ((unsigned*)rec)[lane] = 0u;  // reset for the next round (32 words)
    }
    if (!conf) {
        if (lane == 0) settle(p, io, v, cv);
        maxc = max(maxc, (int)cv);
        return;
    }
    const int ff = window_first_clear(all);
    const uint32_t color = ff >= 0 ? (uint32_t)ff + 1u : rescan_first_fit(p.rowptr, p.colidx, io.Xc, v);
    if (lane < 8u) p.stat[(size_t)v * 8 + lane] = stat;
    if (lane == 0) {
        recolor(p, io, v, color);
        vol += (unsigned)kept;
    }
    warp_append_one(io.next, make_int4(v, b, kept, h.e.w));
}

// The largest power of two (its logarithm) not above `most` that leaves a
// task for each 1 / per_warp entries.  Powers of two and a float reciprocal,
// so that no warp divides: a round of little work would feel it, and any
// value gives the same result.
__device__ __forceinline__ unsigned task_shift(unsigned entries, float per_warp, unsigned most) {
    const unsigned x = min(most, (unsigned)((float)entries * per_warp));
    return x <= 1u ? 0u : 31u - (unsigned)__clz((int)x);
}

__device__ __forceinline__ TaskSplit split_round(const RoundSizes& r, unsigned W) {
    TaskSplit q;
    const float w = 1.f / (float)W;
    // S vertices per task: 32 in a large round, down to kShortPerTaskMin as it
    // leaves fewer than four tasks a warp; a task of 32 short lists walks up to
    // 1024 entries in sequence, which in the last rounds was the longest chain of
    // the round
    const unsigned xs = max(task_shift(r.nS, w / 4.f, 32u), task_shift(kShortPerTaskMin, 1.f, 32u));
    // M vertices per task: up to kMedPerTask, fewer (down to 1) likewise, so that
    // a task's chain of per-vertex reads does not set the round's length
    const unsigned xm = task_shift(r.nM, w / 4.f, kMedPerTask);
    // steps of 16, 8, 4 and 2 vertices of the L2 to L16 tasks: as many as leave a
    // task for every other warp (each task waits for two reads in a row and
    // appends once, so that four tasks a warp, as above, cost more than they even
    // out: R-MAT-G of 1,000,003 vertices with keys 1.87 ms against 1.61; one a
    // warp 1.62)
    const unsigned x2 = task_shift(r.n2, w / 8.f, 2u), x4 = task_shift(r.n4, w / 4.f, 4u);
    const unsigned x8 = task_shift(r.n8, w / 2.f, kMidSteps), x16 = task_shift(r.n16, w, kMidSteps);
    q.spt = 1u << xs;
    q.mpt = 1u << xm;
    q.s2 = 1u << x2;
    q.s4 = 1u << x4;
    q.s8 = 1u << x8;
    q.s16 = 1u << x16;
    q.e0 = r.nHC;
    q.e1 = q.e0 + ((r.nM + q.mpt - 1) >> xm);
    q.e2 = q.e1 + ((r.n16 + 2u * q.s16 - 1) >> (1u + x16));
    q.e3 = q.e2 + ((r.n8 + 4u * q.s8 - 1) >> (2u + x8));
    q.e4 = q.e3 + ((r.nS + q.spt - 1) >> xs);
    q.e5 = q.e4 + ((r.n4 + 8u * q.s4 - 1) >> (3u + x4));
    q.total = q.e5 + ((r.n2 + 16u * q.s2 - 1) >> (4u + x2));
    q.nstat = max(2u, (unsigned)((float)q.total * (.5f * w)));
    return q;
}

// One fused pass over U_k, shared among W warps (this warp is number gw).
// Task t: first the H-bin chunks, then the M-bin entries, up to kMedPerTask
// per task (fewer as the round shrinks), L16 and L8 entries in steps of 2 and 4
// (up to kMidSteps of them a task), the S-bin entries, 32 per task (down to
// kShortPerTaskMin as the round shrinks), then L4 and L2 entries in steps of 8
// and 16 (up to 4 and 2); an S or H task reads at most 1024 entries.  Warp gw
// takes tasks gw, gw + W, ... for half of its even
// share (at least two); then, with a counter (ctr), it claims one task at a
// time (nstat W + the counter's old value), so that warps that drew cheap
// tasks take more and the round ends when the work does, not when the
// unluckiest warp's fixed share does, while only about half the tasks cost an
// atomic on the counter's line; without a counter it keeps taking every W-th
// task.  The next task's head is loaded, and the claim after it issued,
// before the current task runs, so neither waits on memory.
template <typename T, bool P>  // P: a priority array is given
__device__ __forceinline__ void run_pass(const Params<T>& p, int k, const RoundSizes& r, int& maxc, unsigned gw,
                                         unsigned W, unsigned* ctr) {
    __shared__ FlatSmem s_flat[kWarpsPerBlockMax];
    const PassIO<T> io = pass_io(p, k);
    const unsigned wib = threadIdx.x >> 5;
    // the split sits in shared memory: it is the same for every warp, read once a
    // task, and would take some twenty registers across the loop
    __shared__ RoundSizes s_sizes;
    __shared__ TaskSplit s_split;
    if (threadIdx.x == 0) {
        s_sizes = r;
        s_split = split_round(r, W);
    }
    __syncthreads();
    const RoundSizes& z = s_sizes;
    const TaskSplit& q = s_split;
    const unsigned total = q.total;
    unsigned vol = 0;  // this lane's share of the next round's read volume
    // this warp's tasks: gw + jW for j < nstat, then claimed ones from nstat W on
    const unsigned nstat = ctr ? q.nstat : 0xffffffffu;
    TaskHead cur;
    if (gw < total) cur = load_head(io, gw, z, q);
    unsigned tn = gw + W;
    unsigned j = 0;  // position of the current task in that sequence
    for (unsigned t = gw; t < total; ++j) {
        TaskHead nxt;
        if (tn < total) nxt = load_head(io, tn, z, q);
        // the task after next: fixed, or claimed now (its number is needed after this task)
        const bool fixed = j + 2u < nstat;
        unsigned claim = 0;
        if (!fixed && tn < total && lane_id() == 0) claim = atomicAdd(ctr, 1u);
        if (t < q.e0) {
            if (P && io.first) hub_chunk<T, P, P>(p, io, cur, s_flat[wib], maxc, vol);
            else hub_chunk<T, P, false>(p, io, cur, s_flat[wib], maxc, vol);
        } else if (t < q.e1) {
            if (P && io.first) vertex_task<T, P, P>(p, io, cur.e, s_flat[wib], maxc, vol);
            else vertex_task<T, P, false>(p, io, cur.e, s_flat[wib], maxc, vol);
        } else if (t < q.e2) {
            mid_task<T, P, 16>(p, io, cur.e, q.s16, maxc, vol);
        } else if (t < q.e3) {
            mid_task<T, P, 8>(p, io, cur.e, q.s8, maxc, vol);
        } else if (t < q.e4) {
            flat_task<T, P>(p, io, cur.e, s_flat[wib], maxc, vol);
        } else if (t < q.e5) {
            tiny_task<T, P, 4>(p, io, cur.e, q.s4, maxc, vol);
        } else {
            tiny_task<T, P, 2>(p, io, cur.e, q.s2, maxc, vol);
        }
        const unsigned tnn = fixed ? tn + W : nstat * W + __shfl_sync(kFull, claim, 0);
        t = tn;
        cur = nxt;
        tn = tn < total ? tnn : total;
    }
    fold_volume(p.st, p.round_vol, p.round_cap, k + 1, vol);
}

// All rounds k >= 2 in one cooperative launch; a bounded grid barrier
// separates the rounds.  Every block reads the same counts and status after
// a barrier, so all blocks take the same decisions in the same round.  Once a
// round reads at most p.tail_volume entries, block 0 runs the remaining rounds
// alone, separated by block barriers (the other blocks leave): the same
// synchronous rounds, without the cost of a grid barrier per round.
template <typename T, bool P>  // P: a priority array is given
__global__ void __launch_bounds__(256, kMinBlocks) rounds_persistent_kernel(Params<T> p) {
    RoundState* st = p.st;
    int maxc = 0;
    unsigned gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    unsigned W = (gridDim.x * blockDim.x) >> 5;
    bool tail = false;
    for (int k = 2;; ++k) {
        const RoundCounts& c = st->rc[k % 3];
        unsigned size;
        const RoundSizes r = round_sizes_of(c, &size);
        // start of this pass (the last record, for the empty round, marks the end)
        if (p.round_ns && blockIdx.x == 0 && threadIdx.x == 0 && k - 1 <= p.round_cap)
            p.round_ns[k - 1] = globaltimer_ns();
        if (size == 0) {
            if (blockIdx.x == 0 && threadIdx.x == 0) st->rounds = k - 1;
            break;
        }
        // (the word that round k - 1 wrote, not st->status: a block already working
        // on this round may set that, and all blocks have to stop in the same round)
        if (r.overflow) break;
        if (k > p.max_rounds) {
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                st->rounds = k - 1;
                st->status = kStatusMaxRounds;
            }
            break;
        }
        if (!tail && p.tail_volume >= 0 && __ldcg(&st->rc[k % 3].vol) <= (unsigned)p.tail_volume) {
            if (blockIdx.x != 0) break;
            tail = true;
            gw = threadIdx.x >> 5;
            W = blockDim.x >> 5;
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            RoundCounts& z = st->rc[(k + 2) % 3];
            z.overflow = z.s = z.m = z.vol = 0u;
            z.tiny = z.mid = z.hc = 0ull;
            st->task_next[(k + 1) % 3] = 0u;  // round k + 1's claims (no one touches it in round k)
            if (k - 1 < p.round_cap) p.round_sizes[k - 1] = (int32_t)size;
        }
        run_pass<T, P>(p, k, r, maxc, gw, W, &st->task_next[k % 3]);
        if (tail) {
            __threadfence();
            __syncthreads();
        } else if (!grid_barrier(st, p.barrier_polls, (unsigned)k - 2u)) {
            break;
        }
    }
    fold_max_color(st, maxc);
}

// One pass per launch (loop mode 1): counts come from the host.
template <typename T, bool P>  // P: a priority array is given
__global__ void __launch_bounds__(256, kMinBlocks) round_kernel(Params<T> p, int k, RoundSizes r) {
    int maxc = 0;
    run_pass<T, P>(p, k, r, maxc, (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
             (gridDim.x * blockDim.x) >> 5, nullptr);
    fold_max_color(p.st, maxc);
}

// ------------------------------------------------------------ validation

__device__ __forceinline__ uint64_t fmix64(uint64_t k) {
    // MurmurHash3 64-bit finaliser (Appleby)
    k ^= k >> 33;
    k *= 0xff51afd7ed558ccdull;
    k ^= k >> 33;
    k *= 0xc4ceb9fe1a85ec53ull;
    k ^= k >> 33;
    return k;
}

// Loop mode 2: the rounds as a CUDA graph whose while node repeats
// graph_round_kernel + graph_cond_kernel on the device.  graph_round_kernel
// runs round st->graph_round over the counts that the previous pass left.
template <typename T, bool P>  // P: a priority array is given
__global__ void __launch_bounds__(256, kMinBlocks) graph_round_kernel(Params<T> p) {
    RoundState* st = p.st;
    const int k = __ldcg(&st->graph_round);
    // the counts by one thread, which alone splits them into tasks: six words that
    // every warp of the GPU takes from one L2 line each are 2 us of a short round
    RoundSizes r = {};
    unsigned size;
    if (threadIdx.x == 0) r = round_sizes_of(st->rc[k % 3], &size);
    int maxc = 0;
    run_pass<T, P>(p, k, r, maxc, (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
             (gridDim.x * blockDim.x) >> 5, nullptr);
    fold_max_color(st, maxc);
}

// One thread, after round k (k = 1 before the loop): decide whether round k + 1
// runs, clear the counters it will append to, and set the while condition.
template <typename T>
__global__ void graph_cond_kernel(Params<T> p, int before_loop, cudaGraphConditionalHandle handle) {
    RoundState* st = p.st;
    const int k = before_loop ? 1 : st->graph_round;
    const int kn = k + 1;
    const RoundCounts& c = st->rc[kn % 3];
    const unsigned size = low_count(c.tiny) + high_count(c.tiny) + low_count(c.mid) + high_count(c.mid) + c.s + c.m +
                          hub_count(c.hc);
    unsigned go = 0u;
    if (size == 0u) {
        st->rounds = k;
    } else if (st->status == kStatusColorOverflow) {
        st->rounds = k;
    } else if (kn > p.max_rounds) {
        st->rounds = k;
        st->status = kStatusMaxRounds;
    } else {
        RoundCounts& z = st->rc[(kn + 1) % 3];
        z.overflow = z.s = z.m = z.vol = 0u;
        z.tiny = z.mid = z.hc = 0ull;
        if (kn - 1 < p.round_cap) p.round_sizes[kn - 1] = (int32_t)size;
        st->graph_round = kn;
        go = 1u;
    }
    __threadfence();
    cudaGraphSetConditional(handle, go);
}

struct ValidateOut {
    unsigned long long asym;  // 0 when the entries are symmetric
    int bad_index, self_loop;
};

// What entry w of row v adds to ValidateOut::asym: a hash of the pair {v, w},
// with the sign of its direction, so that an edge present in both directions
// (equally often) cancels out and any other leaves a sum that is 0 with a
// probability of about 2^-64.
__device__ __forceinline__ uint64_t asymmetry(int32_t v, int32_t w) {
    const uint32_t lo = (uint32_t)min(v, w), hi = (uint32_t)max(v, w);
    const uint64_t h = fmix64(((uint64_t)lo << 32) | hi);
    return v < w ? h : 0ull - h;
}

// Range, self-loop and symmetry checks of every entry.  A warp takes up to 32
// rows: those of up to kPass1Flat entries are read as one flat, coalesced range,
// longer ones by the whole warp in turn, and those above kCheckFar by the whole
// block when its warps are done with the others.  Fewer rows (a power of two) when that
// would leave warps without any, as long as they hold 128 entries, so that a
// graph of few long rows is spread over the GPU.  Runs behind the setup scan and
// does nothing when that found the row starts unusable.
//
// Bound: the hash, some 25 instructions an entry; the entries are read once.  A
// warp per row (4 of 32 lanes on a mesh), two hashes an entry and two global
// atomics a thread, waited for on its own, cost 0.17 ms more on the 4.0 M
// entries of a 997,399-vertex mesh (a checked call 0.42 ms, now 0.26).  With 32
// rows always, K(2000, 2000), 4,000 rows of 2,000 entries, took 217 us, now 20;
// G(3000, 12000) 4.3, now 3.7; G(400000, 6000000) 38.9, now 37.0.  With the
// longest rows left to a warp, K(2, 200000) took 1,179 us, now 151, and a star of
// 1M vertices 2,964, now 380.
constexpr int kCheckFar = 8192, kCheckFarRows = 64;
__global__ void __launch_bounds__(256) validate_kernel(const int32_t* __restrict__ rowptr,
                                                       const int32_t* __restrict__ colidx, int32_t n,
                                                       const Stats* __restrict__ scan, ValidateOut* out) {
    struct Smem {
        uint8_t lane_of[32];  // lane of the i-th non-empty row
    };
    __shared__ Smem s_row[8];
    __shared__ unsigned long long s_sum[8];
    __shared__ int32_t s_far[kCheckFarRows];  // rows for the whole block
    __shared__ int s_nfar;
    // (read through L1: a word that every warp of the GPU takes from L2 costs 4 us)
    const int bad_rows = __ldg(&scan->bad), nnz = __ldg(&scan->nnz);
    if (bad_rows || nnz < 0 || (nnz > 0 && !colidx)) return;
    if (threadIdx.x == 0) s_nfar = 0;
    __syncthreads();
    const unsigned lane = lane_id(), wib = threadIdx.x >> 5;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t W = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const float most = fmaxf((float)n / (float)W, 128.f * (float)n / (float)max(nnz, 1));
    const int shift = 31 - __clz((int)fminf(32.f, fmaxf(1.f, most))), rows = 1 << shift;
    const int64_t ntasks = ((int64_t)n + rows - 1) >> shift;
    const uint64_t pol = policy_evict_first();
    uint64_t sum = 0;
    bool bad = false, loop = false;
    auto entry = [&](int32_t v, int32_t w) {
        if ((uint32_t)w >= (uint32_t)n) {
            bad = true;
        } else {
            loop |= w == v;
            sum += asymmetry(v, w);
        }
    };
    // entries [i, e) of row v, from i on every `step`-th group of 256
    auto entries = [&](int32_t v, int64_t i, int64_t e, int step) {
        for (i += lane; i < e; i += step) {
            int32_t w[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) w[u] = i + 32 * u < e ? ld_adj(colidx + i + 32 * u, pol) : 0;
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (i + 32 * u < e) entry(v, w[u]);
        }
    };
    for (int64_t t = gw; t < ntasks; t += W) {
        const int64_t vv = (t << shift) + lane;
        const bool valid = (int)lane < rows && vv < n;
        const int32_t v = valid ? (int32_t)vv : 0;
        const int32_t b = valid ? __ldg(rowptr + v) : 0;
        const int32_t d = valid ? __ldg(rowptr + v + 1) - b : 0;
        const int32_t eff = d > kPass1Flat ? 0 : d;
        int32_t incl = eff;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t x = __shfl_up_sync(kFull, incl, o);
            if ((int)lane >= o) incl += x;
        }
        const int32_t off = incl - eff;
        const int32_t D = __shfl_sync(kFull, incl, 31);
        const unsigned nz = __ballot_sync(kFull, eff > 0);
        if (eff > 0) s_row[wib].lane_of[__popc(nz & ((1u << lane) - 1u))] = (uint8_t)lane;
        const int32_t b_off = b - off;
        __syncwarp();
        for (int32_t F0 = 0; F0 < D; F0 += 32 * 4) {
            int32_t w[4], own[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int32_t base = F0 + 32 * u;
                const int32_t f = base + (int32_t)lane;
                const int32_t rel = off - base;
                const unsigned before = __popc(__ballot_sync(kFull, eff > 0 && rel < 0));
                const unsigned starts = __reduce_or_sync(kFull, (eff > 0 && rel >= 0 && rel < 32) ? (1u << rel) : 0u);
                const unsigned rank = before + __popc(starts & (0xffffffffu >> (31 - lane)));
                own[u] = (f < D && rank > 0) ? (int)s_row[wib].lane_of[rank - 1] : 0;
                const int32_t rb = __shfl_sync(kFull, b_off, own[u]);
                w[u] = f < D ? ld_adj(colidx + rb + f, pol) : 0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (F0 + 32 * u + (int32_t)lane < D) entry((int32_t)(t << shift) + own[u], w[u]);
        }
        bool later = false;
        if (d > kCheckFar) {
            const int at = atomicAdd(&s_nfar, 1);
            later = at < kCheckFarRows;
            if (later) s_far[at] = v;
        }
        unsigned big = __ballot_sync(kFull, d > kPass1Flat && !later);
        while (big) {
            const int j = __ffs(big) - 1;
            big &= big - 1;
            const int64_t bj = __shfl_sync(kFull, b, j);
            entries((int32_t)(t << shift) + j, bj, bj + __shfl_sync(kFull, d, j), 256);
        }
        __syncwarp();
    }
    __syncthreads();
    for (int j = 0; j < min(s_nfar, kCheckFarRows); ++j) {
        const int32_t v = s_far[j];
        entries(v, (int64_t)__ldg(rowptr + v) + 256 * wib, __ldg(rowptr + v + 1), 256 * (int)(blockDim.x / 32));
    }
    if (__any_sync(kFull, bad) && lane == 0) out->bad_index = 1;
    if (__any_sync(kFull, loop) && lane == 0) out->self_loop = 1;
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
    if (lane == 0) s_sum[wib] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (unsigned i = 1; i < blockDim.x / 32; ++i) sum += s_sum[i];
        if (sum) atomicAdd(&out->asym, (unsigned long long)sum);
    }
}

}  // namespace gc
