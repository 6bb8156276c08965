// Level-synchronous batch peeling through the BE-Index (Section V-B,
// Alg. 5, BiT-BU++; the <= k frontier rule of Alg. 4).
//
// One round removes the batch S = {unassigned e : support(e) <= k} at once:
//   kills (Alg. 5, the loop over e in S and B in N_I(e)):
//     every live twin pair of a bloom B that holds an edge of S dies once;
//     C(B) counts the dead pairs.  When both twins are in S the pair is
//     counted once (the example of Section V-B: three twin pairs of B0 drop
//     its bloom number to 0).  A twin outside S loses all k_B - 1
//     butterflies it had in B (Lemma 2).
//   bloom phase (Alg. 5, the loop over blooms with C(B) > 0):
//     every edge of a surviving pair of B loses C(B) butterflies (one per
//     dead pair); then k_B -= C(B), so the bloom keeps C(k_B - C, 2)
//     butterflies (Lemma 1).
//   phi(e) = k for e in S.
// k only grows: when no unassigned edge has support <= k, k jumps to the
// minimum remaining support (the batch-edge rule of Lemma 9).  Supports are
// decremented without the max(MBS, .) clamp of Alg. 5; an edge that drops to
// or below k is taken by the next round with the same k, which gives the same
// phi.  An edge joins the next batch exactly when one decrement carries its
// support from above k to <= k, so rounds inside a level never rescan edges.
//
// Scheduling.  The whole loop runs in one persistent cooperative kernel (one
// block per SM slot the occupancy allows); phases are separated by a grid
// barrier whose wait is bounded by a timer (on timeout the kernel raises an
// error word and every block returns).  The kills of round r + 1 need only
// C_r, which is final once the bloom phase of round r starts, so they are
// made inside that bloom phase: the warp whose decrement carries an edge
// into the batch of round r + 1 kills the edge's twin pairs at once when the
// edge has few links, and queues the links as incidence items otherwise.  A
// round therefore costs one barrier, plus a separate incidence phase (and a
// second barrier) only when such items exist or a level jump selected the
// batch.  Pairs killed early carry stamp r + 1 and still count as alive in
// the bloom phase of round r.  The bloom number at the start of round q is
// the value recorded after the last round before q that touched the bloom; the
// bloom's first item of round q records the new one during q's bloom phase.
// Work is split into items of at most kSeg entries, so no warp straggles on a
// hub edge or bloom; a warp lays the entries of its items side by side.  A twin
// pair carries the round it died in; the edges of a batch race to stamp it with
// atomicCAS, so exactly one of them counts it in C(B); the stamp also records
// which members of the pair are in the batch (the killer's side bit, and the
// other member's bit when it stamps the same round), so the bloom phase knows
// which member loses k_B - 1 without reading edge states.  Counters and work lists
// rotate by round (C by 3, bloom items by 4, batch sizes by 3, incidence items
// by 2) so each is reset a barrier after its last reader.  Data written by other blocks
// during the kernel is read with L2 (.cg) loads.
//
// Coarse peel (kCoarse).  The same rounds with levels that are ranges of bitruss
// numbers: a level takes every edge whose support is, or falls, within the range,
// so phi is known only up to the range (the part), in a fraction of the rounds
// (2M-edge graph: 865 instead of 39,928).  Each part can then be peeled by itself
// (split.cu, local.cu).  A level jump reads the alive edges, copies their
// supports, histograms them by class and takes classes until their weight (edges
// and links) reaches the target; a graph that parts do not suit is given up at the
// first one (kNarrow).  The jump's list of alive edges is written
// anew only after a quarter has gone: taking places from one counter at every
// jump cost 130 us of it at 2M edges (now 23 us).  What bounds it are the bloom
// phases (31 of 41 ms at 2M edges, 45 of 59 with planted bicliques): 1.2 G pair
// slots at 38 G a second, scattered loads and atomics through L2; on 76 of the
// 152 SMs the peel takes 1 % longer at 200,000 edges, on 16 a third.
#include <limits.h>
#include <stddef.h>

#include "bt_device.cuh"
#include "bt_internal.cuh"

namespace bt {
namespace {

// entries per work item: SEG = 32, 64 or 128 (template parameter: 32 or 64
// picked by the batch autotuner, 128 for indexes of over 2^30 twin pairs;
// a coarse peel knows 32 and 128).  Threads a block: 640 (96 registers, no spills) for 32- and
// 64-entry items, 512 (128 registers) for 128-entry items, whose four slots
// a lane need the registers.
__host__ __device__ constexpr int peel_threads(uint32_t seg) { return seg == 128 ? 512 : 640; }
// Lane l of warp w takes item w + l * nwarps (plus multiples of 32 * nwarps),
// and the warp works on the entries of its items side by side: a round with
// fewer items than warps still gives every item its own warp, and a large
// round fills all lanes however small its items are.
// edges that join the next batch in a bloom phase are listed per block (up to
// one per thread); the block kills their twin pairs at the end of the phase,
// two links per thread, for the edges whose links fit in the first two per
// thread
constexpr unsigned long long kBarrierTimeoutNs = 20ull * 1000 * 1000 * 1000;  // 20 s (default)
// pair death stamps: round << 2 | (first member in the batch) | (second << 1);
// kAlive (all ones) is never a stamp while rounds stay below kMaxRounds
constexpr uint32_t kMaxRounds = (1u << 30) - 4u;
constexpr uint32_t kErrBarrier = 1u;
constexpr uint32_t kErrRounds = 2u;
constexpr uint32_t kErrPeelOverflow = 4u;
constexpr unsigned kFull = 0xffffffffu;
// level-jump windows above this size queue their batch with warp-aggregated atomics
constexpr uint32_t kWarpSlotsMin = 1u << 16;

// Support classes of the coarse peel: values below 64 apart, above that 64 a
// power of two.
constexpr uint32_t kBins = 2048;
__device__ __forceinline__ uint32_t bin_of(unsigned long long s) {
    if (s < 64ull) return (uint32_t)s;
    const uint32_t x = s > 0x7FFFFFFFull ? 0x7FFFFFFFu : (uint32_t)s;
    const uint32_t e = 31u - (uint32_t)__clz(x);
    return ((e - 5u) << 6) + ((x >> (e - 6u)) & 63u);
}
__device__ __forceinline__ long long bin_top(uint32_t b) {
    if (b < 64u) return b;
    const uint32_t e = (b >> 6) + 5u;
    return ((long long)(64u + (b & 63u) + 1u) << (e - 6u)) - 1;
}

// Parts pay where bitruss numbers spread: many levels, and ranges of a few per cent
// of the links each.  Where the supports lie close together (dense blocks,
// uniform random graphs) almost all edges go in one avalanche: few rounds, each of
// them wide enough for the grid, and one range with nearly everything in it, which
// a block or a cluster would peel by itself.  Supports tell: of the links, the
// share on edges within a factor of 8 in support was 0.957 on a random graph of mean
// degree 25, 1.0 on denser ones, blocks and equal bicliques, 0.29 to 0.67 on skewed graphs
// of 1,000 to 30M edges, 0.89 and 0.95 on ones with a single dominating block.  From
// kNarrow on the grid peels the whole graph (by parts instead: a random
// graph of 2M edges, mean degree 100, 62 ms against 19; a block of 300 x 300 of
// density 0.9, 14.1 against 2.2; K_{200,200} 10.9 against 0.3).
constexpr float kNarrow = 0.955f;
// Nor do parts pay where hardly any edge has a support above kLow: there are no more
// levels than that below it, and a rest of kRest links has few rounds (82 at 24,000).
// A random graph of 100,000 edges (mean degree 25, 0.957 as above) 1.26 ms by parts,
// 0.41 by the grid; 1M edges with a light tail 0.96 and 0.5.
constexpr uint32_t kLow = 24, kRest = 1u << 14;

struct Ctl {
    unsigned long long bar_count;  // barrier arrivals (monotonic within a launch)
    unsigned int err;
    unsigned int pad0;
    unsigned int n_items[2];  // incidence items, by round parity
    unsigned int n_edges[3];  // batch sizes, by round mod 3
    unsigned int n_bseg[4];   // bloom items, by round mod 4
    unsigned int n_alive[2];  // alive list sizes (ping-pong)
    unsigned int n_near[2];   // near-window list sizes (ping-pong)
    unsigned int pad1;
    unsigned long long minsup;   // level-jump minimum over the near window
    unsigned long long minsup2;  // minimum over all alive edges (window rebuild)
    unsigned long long updates;
    unsigned long long slots;  // bloom pair slots visited by the bloom phase
    unsigned long long scanned;  // edge-list entries scanned by level jumps
    unsigned long long rounds;
    unsigned long long levels;
    unsigned long long windows;
    unsigned long long kfinal;
    unsigned long long inc_phases;  // rounds that ran a separate incidence phase
    unsigned int n_parts;           // coarse peel: parts made
    unsigned int narrow;            // coarse peel: given up, the supports lie close together
    unsigned int n_zero;            // coarse peel: edges without butterflies, part 0
    unsigned long long first_rounds, first_levels, first_updates;  // of its first part, with k_init
    unsigned int hist[2][kBins];    // coarse peel: supports of the alive edges, ping-pong
};

// What changes of a bloom, in one 32-byte sector.  A kill touches it with one
// counter atomic and no load: a load beside an atomic on the same sector
// costs three times the atomic (the part peel's kills went from 14 to 5 ns
// a link an SM without it).
struct __align__(32) BloomWord {
    unsigned long long bw;      // last round that touched it << 32 | k_B after it
    uint32_t C[3];              // C_r by round mod 3
    uint32_t pad[3];
};

struct PeelArgs {
    uint64_t m;
    const uint64_t *inc_off;
    const uint2 *inc;  // (pair, bloom | side << 31)
    const uint2 *pairs;
    const uint32_t *bloom_off;
    BloomWord *blooms;
    int *sup;  // below m < 2^31: k butterflies on an edge need k other edges opposite it
    uint32_t *state;
    uint32_t *phi;
    uint32_t *died;           // death stamp of a twin pair (kAlive while alive)
    uint4 *items[2];          // (edge, first link lo, first link hi, count | head flag << 31)
    uint4 *bseg[4];           // (bloom, first pair, count | head flag << 31, 0)
    uint32_t *alive[2];
    uint32_t *near[2];
    uint64_t item_cap;
    uint64_t bseg_cap;
    Ctl *ctl;
    uint64_t round_limit;
    unsigned long long barrier_timeout_ns;
    unsigned long long hold_barrier;  // 0, or n: block 0 skips its arrival at barrier n (from 1)
    uint32_t join_cap;     // edges a block lists in a bloom phase (<= threads a block)
    uint32_t block_links;  // links of the listed edges the block stage kills itself (<= 2 a thread)
    // progressive compression: peel only the m_active unassigned edges, start
    // at level k_init, and record phi only for levels >= assign_from
    uint64_t m_active;
    long long k_init;
    long long assign_from;
    // coarse peel: phi receives the part of every edge instead, snap its support
    // when its part began.  An edge weighs 1 + (links >> wshift), a part aims at
    // a weight of `target`.
    int *snap;
    uint32_t target, wshift;
    uint32_t max_parts;
};

// Loop state every thread keeps identically (derived from values read after
// grid barriers).
struct Lvl {
    long long k;    // current level
    long long khi;  // top of the near window: alive edges with support < khi are listed
    uint32_t nq;    // current near list
    uint32_t label;  // what a peeled edge receives: k, or its part in a coarse peel
};

__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t ldcg_u32(const uint32_t *p) { return __ldcg(p); }
__device__ __forceinline__ long long ldcg_ll(const int *p) { return __ldcg(p); }

// Grid-wide barrier over all blocks of a cooperative launch.  Arrivals go
// to one monotonic counter (release); barrier number b completes when the
// counter reaches (b + 1) * gridDim.x, which every block polls (acquire).
// Returns false when the wait timed out or another block raised an error.
__device__ __forceinline__ void arrive_release(unsigned long long *p) {
    asm volatile("red.release.gpu.global.add.u64 [%0], 1;" ::"l"(p) : "memory");
}
__device__ __forceinline__ unsigned long long load_acquire(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Counters the next phase needs.  Thread 0 of each block reads them once
// after the barrier and hands them to its block through shared memory, so a
// counter that every thread needs costs one L2 request per block instead of
// one per warp (same-address requests queue up at one L2 slice).
struct Snap {
    const unsigned int *u[5];
    const unsigned long long *w;
};
struct SnapVals {
    unsigned int u[5];
    unsigned long long w;
};

__device__ bool grid_barrier(const PeelArgs &a, unsigned long long &bar_no, const Snap &sn, SnapVals *s_v) {
    Ctl *ctl = a.ctl;
    __syncthreads();
    __shared__ int s_ok;
    const unsigned long long target = (bar_no + 1) * gridDim.x;
    ++bar_no;
    if (threadIdx.x == 0) {
        int ok = 1;
        // a held barrier (fault injection) never completes: every block's
        // wait below runs out and raises the error word
        if (!(blockIdx.x == 0 && bar_no == a.hold_barrier)) arrive_release(&ctl->bar_count);
        if (load_acquire(&ctl->bar_count) < target) {
            const unsigned long long t0 = now_ns();
            unsigned int spins = 0;
            while (load_acquire(&ctl->bar_count) < target) {
                if (((++spins) & 63u) == 0) {
                    if (*(volatile unsigned int *)&ctl->err) {
                        ok = 0;
                        break;
                    }
                    if (now_ns() - t0 > a.barrier_timeout_ns) {
                        atomicOr(&ctl->err, kErrBarrier);
                        ok = 0;
                        break;
                    }
                }
            }
        }
        if (ok) {
            unsigned int v[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) v[i] = sn.u[i] ? __ldcg(sn.u[i]) : 0u;
            const unsigned long long w = sn.w ? __ldcg(sn.w) : 0ull;
#pragma unroll
            for (int i = 0; i < 5; ++i) s_v->u[i] = v[i];
            s_v->w = w;
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Queue the links [ib, ie) of edge e as incidence items of list dst, one item
// per kSeg links, each carrying its link range.
template <uint32_t kSeg>
__device__ __forceinline__ void push_items(const PeelArgs &a, uint32_t e, uint32_t dst, uint64_t ib,
                                           uint64_t ie) {
    const uint64_t d = ie - ib;
    if (d == 0) return;
    const uint32_t nseg = (uint32_t)((d + kSeg - 1) / kSeg);
    const uint32_t base = atomicAdd(&a.ctl->n_items[dst], nseg);
    for (uint32_t s = 0; s < nseg; ++s) {
        const uint64_t j = ib + (uint64_t)s * kSeg;
        const uint64_t left = d - (uint64_t)s * kSeg;
        const uint32_t cnt = (uint32_t)(left < kSeg ? left : kSeg);
        a.items[dst][base + s] =
            make_uint4(e, (uint32_t)j, (uint32_t)(j >> 32), cnt | (s == 0 ? 0x80000000u : 0u));
    }
}

// Edge e joins the batch of round q at level k.
__device__ __forceinline__ void join_batch(const PeelArgs &a, uint32_t e, uint32_t q, const Lvl &L) {
    a.state[e] = q;
    if (L.k >= a.assign_from) a.phi[e] = L.label;  // e leaves in a batch of this level
}

__device__ __forceinline__ void push_near(const PeelArgs &a, uint32_t e, uint32_t nq) {
    a.near[nq][atomicAdd(&a.ctl->n_near[nq], 1u)] = e;
}

// Window above the current minimum: narrow enough that a level jump scans few
// edges at high levels (dense cores hold many edges in a support range), wide
// enough that rebuilds from the full alive list stay rare.
__device__ __forceinline__ long long window_top(long long kmin) {
    long long w = kmin / 64;
    return kmin + (w < 8 ? 8 : w);
}

// Edges of the batch of round q kill the pairs of up to N links (won[r] set
// on entry for the valid ones; link l[r] names the pair and which member the
// edge is, 0 first, 1 second).  The first edge to stamp a pair counts it
// (won[r] stays true); a twin of the same batch adds its side bit to the
// stamp.  A lane's stamps go out together before any result is examined.
template <uint32_t N>
__device__ __forceinline__ void kill_pairs(const PeelArgs &a, const uint2 (&l)[N], bool (&won)[N], uint32_t q) {
    uint32_t old[N];
#pragma unroll
    for (uint32_t r = 0; r < N; ++r)
        old[r] = won[r] ? atomicCAS(&a.died[l[r].x], kAlive, (q << 2) | (1u << (l[r].y >> 31))) : 0u;
#pragma unroll
    for (uint32_t r = 0; r < N; ++r) {
        if (!won[r]) continue;
        won[r] = old[r] == kAlive;
        if (!won[r] && (old[r] >> 2) == q) atomicOr(&a.died[l[r].x], 1u << (l[r].y >> 31));
    }
}

// Places of bloom items a warp has taken from the list's counter and not filled
// yet: in an incidence phase a warp takes kTake at a time, since millions of
// first kills would otherwise queue on the one counter (about 4 ns each).
// All of them are filled before more are taken, so the list needs room for one
// stock a warp beside its items; what is left at the end is filled with empty items.
constexpr uint32_t kTake = 128;
struct Slots {
    uint32_t next = 0, left = 0;
};
__device__ __forceinline__ void fill_empty(const PeelArgs &a, uint32_t qb, Slots &t, int lane) {
    for (uint32_t i = lane; i < t.left; i += 32) a.bseg[qb][t.next + i] = make_uint4(0u, 0u, 0u, 0u);
    t.left = 0;
}

// Whole warp (converged): each lane's pairs killed for round q (won[r], bloom
// B[r]) are counted, and the blooms killed for the first time in round q get
// their bloom items (one per kSeg pairs).  kMode: how the places of the items
// are taken: 0 one counter atomic a warp, 1 one a block (called by the whole
// block), 2 from the warp's stock t.
template <uint32_t kSeg, uint32_t N, int kMode>
__device__ __forceinline__ void warp_kills(const PeelArgs &a, uint32_t q, const uint32_t (&B)[N],
                                           const bool (&won)[N], int lane, Slots &t) {
    // a lane's loads, then its counter atomics, go out together
    uint32_t bo0[N], span[N], prev[N], nseg[N];
    uint32_t mine = 0;
#pragma unroll
    for (uint32_t r = 0; r < N; ++r) {
        bo0[r] = won[r] ? a.bloom_off[B[r]] : 0u;
        span[r] = won[r] ? a.bloom_off[B[r] + 1] - bo0[r] : 0u;
    }
#pragma unroll
    for (uint32_t r = 0; r < N; ++r) prev[r] = won[r] ? atomicAdd(&a.blooms[B[r]].C[q % 3u], 1u) : 1u;
#pragma unroll
    for (uint32_t r = 0; r < N; ++r) {
        nseg[r] = prev[r] == 0u ? (span[r] + kSeg - 1) / kSeg : 0u;
        mine += nseg[r];
    }
    const uint32_t qb = q & 3u;
    uint32_t slot, cut = 0xFFFFFFFFu, jump = 0;  // places from `cut` on lie `jump` further
    if constexpr (kMode == 1) {
        uint32_t all;
        slot = dev::block_excl_scan<uint32_t>(mine, &all);
        if (all == 0) return;
        __shared__ uint32_t s_base;
        if (threadIdx.x == 0) s_base = atomicAdd(&a.ctl->n_bseg[qb], all);
        __syncthreads();
        slot += s_base;
    } else {
        const uint32_t incl = dev::warp_incl_scan(mine);
        const uint32_t all = __shfl_sync(kFull, incl, 31);
        if (all == 0) return;
        if constexpr (kMode == 2) {
            slot = t.next + incl - mine;
            if (all > t.left) {
                const uint32_t more = all - t.left, take = more > kTake ? more : kTake;
                uint32_t base = 0;
                if (lane == 0) base = atomicAdd(&a.ctl->n_bseg[qb], take);
                base = __shfl_sync(kFull, base, 0);
                cut = t.next + t.left;
                jump = base - cut;
                t.next = base + more;
                t.left = take - more;
            } else {
                t.next += all;
                t.left -= all;
            }
        } else {
            uint32_t base = 0;
            if (lane == 31) base = atomicAdd(&a.ctl->n_bseg[qb], all);
            slot = __shfl_sync(kFull, base, 31) + incl - mine;
        }
    }
#pragma unroll
    for (uint32_t r = 0; r < N; ++r)
        for (uint32_t s = 0; s < nseg[r]; ++s, ++slot) {
            const uint32_t left = span[r] - s * kSeg;
            a.bseg[qb][kMode == 2 && slot >= cut ? slot + jump : slot] =
                make_uint4(B[r], bo0[r] + s * kSeg, (left < kSeg ? left : kSeg) | (s == 0 ? 0x80000000u : 0u), 0u);
        }
}

// Edge e joins the batch of round q in a bloom phase: it goes to the block's
// list, or, when that is full, the lane queues its links itself.
template <uint32_t kSeg>
__device__ __forceinline__ void join_next(const PeelArgs &a, uint32_t e, uint32_t q, const Lvl &L,
                                          uint32_t *s_je, uint32_t *s_jn) {
    const uint32_t slot = atomicAdd(s_jn, 1u);
    if (slot < a.join_cap) {
        s_je[slot] = e;
    } else {
        join_batch(a, e, q, L);
        push_items<kSeg>(a, e, q & 1u, a.inc_off[e], a.inc_off[e + 1]);
        atomicAdd(&a.ctl->n_edges[q % 3u], 1u);
    }
}

// Bloom phase of round r, N pair slots (died stamps d, members pr) of a bloom
// with c pairs killed this round and bloom number kB at round start.  All the
// slots' support decrements are issued before any result is examined, so they
// travel together.
template <uint32_t kSeg, uint32_t N>
__device__ __forceinline__ void apply_slots(const PeelArgs &a, const uint32_t (&d)[N], const uint2 (&pr)[N],
                                            const uint32_t (&c)[N], const uint32_t (&kB)[N], const Lvl &L,
                                            uint32_t round, unsigned long long &upd, uint32_t *s_je, uint32_t *s_jn) {
    const uint32_t q = round + 1u;
    uint32_t e[2 * N];
    int dec[2 * N];
#pragma unroll
    for (uint32_t r = 0; r < N; ++r) {
        // bit 31 flags an edge whose bitruss number is already known: it is
        // never peeled again, so it needs no decrement
        const bool fx = pr[r].x >> 31, fy = pr[r].y >> 31;
        e[2 * r] = pr[r].x & 0x7FFFFFFFu;
        e[2 * r + 1] = pr[r].y & 0x7FFFFFFFu;
        dec[2 * r] = 0;
        dec[2 * r + 1] = 0;
        const uint32_t dr = d[r] >> 2;  // round of death (kAlive: 0x3FFFFFFF, no round)
        if (d[r] == kAlive || dr == q) {
            // alive during this round (a pair killed for the next round still
            // is): one butterfly lost per dead pair
            if (!fx) dec[2 * r] = c[r];
            if (!fy) dec[2 * r + 1] = c[r];
        } else if (dr == round && kB[r] > 1u) {
            // died now: a member outside S (its bit not stamped) loses its
            // k_B - 1 butterflies
            if (!(fx || (d[r] & 1u))) dec[2 * r] = (int)kB[r] - 1;
            if (!(fy || (d[r] & 2u))) dec[2 * r + 1] = (int)kB[r] - 1;
        }
    }
    int old[2 * N];
#pragma unroll
    for (uint32_t i = 0; i < 2 * N; ++i) old[i] = dec[i] ? atomicSub(&a.sup[e[i]], dec[i]) : 0;
#pragma unroll
    for (uint32_t i = 0; i < 2 * N; ++i) {
        if (!dec[i]) continue;
        ++upd;
        const int now = old[i] - dec[i];
        if (old[i] >= L.khi && now < L.khi) push_near(a, e[i], L.nq);
        // exactly one decrement takes the edge from > k to <= k: it joins the
        // next batch
        if (old[i] > L.k && now <= L.k) join_next<kSeg>(a, e[i], q, L, s_je, s_jn);
    }
}

template <uint32_t kSeg, bool kCoarse>
__global__ void __launch_bounds__(peel_threads(kSeg), 1) k_peel(PeelArgs a) {
    constexpr uint32_t R = kSeg / 32;  // entries per lane
    constexpr uint32_t kT = peel_threads(kSeg);
    constexpr uint32_t kJoinCap = kT;
    const int lane = threadIdx.x & 31;
    const uint32_t gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t gtid = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t nthreads = gridDim.x * blockDim.x;
    Ctl *ctl = a.ctl;
    const uint32_t n_zero = kCoarse ? ctl->n_zero : 0u;
    uint64_t remaining = a.m_active - n_zero;
    uint32_t round = 0;
    // (a coarse peel keeps no window: khi below every support)
    Lvl L{a.k_init, kCoarse ? LLONG_MIN : 0ll, 0, (uint32_t)a.k_init};
    uint32_t ap = 0;  // current alive list
    bool level_jump = true;
    unsigned long long upd = 0, slots = 0;
    unsigned long long bar_no = 0;  // barriers passed (identical in every block)
    // edges this block's bloom items carried into the next batch
    __shared__ uint32_t s_je[kJoinCap], s_joff[kJoinCap], s_jd[kJoinCap];
    __shared__ unsigned long long s_jib[kJoinCap];
    __shared__ uint32_t s_jn;
    __shared__ SnapVals s_v;
    __shared__ uint32_t s_hist[kCoarse ? kBins : 1];
    __shared__ uint32_t s_bin, s_cum;
    // coarse: parts begun, the weight the last one began with, all weight then
    uint32_t pno = 0, picked = 1, total_jump = 0;
    float aim = (float)a.target;
    // part 0 may be given (k_init > 0: what lies up to k_init; else the edges without
    // butterflies, if any); the parts whose tops are chosen here follow
    bool in_first = kCoarse && a.k_init > 0;
    const uint32_t first_free = in_first || n_zero ? 1u : 0u;
    bool narrow = false;
    pno = first_free;
    uint32_t hno = 0;                  // level jumps
    long long first_top = LLONG_MIN, lim = 0;  // the first part's window, what a jump takes
    if (threadIdx.x == 0) s_jn = 0;
    __syncthreads();
    // list sizes, kept identically by every thread from the barrier snapshots
    uint32_t v_near = 0;                      // near list L.nq
    uint32_t v_alive = (uint32_t)a.m;         // alive list ap
    uint32_t n_batch = 0, n_items = 0;        // this round's batch and incidence items
    uint32_t nb_cur = 0, nb_prev = 0;         // bloom items of this round and of the last

    while (remaining > 0) {
        const uint32_t par = round & 1u;
        const uint32_t c3 = round % 3u;
        const uint32_t b4 = round & 3u;
        const uint32_t bp = (round + 3u) & 3u;  // previous round's bloom items
        if (round > a.round_limit) {
            if (gtid == 0) atomicOr(&ctl->err, kErrRounds);
            break;
        }
        if constexpr (kCoarse) {
            if (level_jump) {
                // The first part of a given top k_init: the batches are those of the
                // fine peel, whose level jumps take what its window lists.  While
                // the least support is within it, a jump is one reading for the
                // minimum and one for the batch.
                bool within = false;
                if (in_first) {
                    unsigned long long least = ~0ull;
                    for (uint32_t i = gtid; i < v_alive; i += nthreads) {
                        const uint32_t e = ldcg_u32(&a.alive[ap][i]);
                        const uint32_t stv = ldcg_u32(&a.state[e]);
                        const unsigned long long sv = (unsigned long long)ldcg_ll(&a.sup[e]);
                        if (stv == kAlive && sv < least) least = sv;
                    }
                    if (gtid == 0) atomicAdd(&ctl->scanned, (unsigned long long)v_alive);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const unsigned long long y = __shfl_xor_sync(kFull, least, o);
                        least = y < least ? y : least;
                    }
                    if (lane == 0 && least != ~0ull) atomicMin(&ctl->minsup, least);
                    const Snap sn{{nullptr, nullptr, nullptr, nullptr, nullptr}, &ctl->minsup};
                    if (!grid_barrier(a, bar_no, sn, &s_v)) break;
                    const long long mn = (long long)s_v.w;
                    within = mn <= a.k_init;
                    if (within) {
                        if (mn >= first_top) first_top = window_top(mn);
                        L.k = a.k_init;
                        lim = first_top <= a.k_init ? first_top - 1 : L.k;
                        L.label = 0;
                        if (gtid == 0) ++ctl->first_levels;
                    } else {
                        in_first = false;
                        upd = dev::warp_sum(upd);
                        if (lane == 0 && upd) atomicAdd(&ctl->first_updates, upd);
                        upd = 0;
                        if (gtid == 0) ctl->first_rounds = round;
                    }
                }
                constexpr uint32_t U = 4;  // entries a lane has in flight
                if (!within || hno == 0) {
                    // C1: the alive edges again, with their supports' histogram and
                    // a copy of each support (the last copy an edge gets is its
                    // support when its part begins)
                    for (uint32_t i = threadIdx.x; i < kBins; i += kT) s_hist[i] = 0;
                    __syncthreads();
                    if (gtid == 0) atomicAdd(&ctl->scanned, 2ull * v_alive);
                    // the list is written anew only once a quarter of it is gone:
                    // its places come from one counter, which is what that costs
                    const bool anew = remaining < v_alive - v_alive / 4u;
                    for (uint32_t i0 = gwarp * 32u * U; i0 < v_alive; i0 += nthreads * U) {
                        uint32_t e[U], stv[U];
                        long long sv[U];
                        bool keep[U];
#pragma unroll
                        for (uint32_t r = 0; r < U; ++r) {
                            const uint32_t i = i0 + 32u * r + lane;
                            keep[r] = i < v_alive;
                            e[r] = keep[r] ? ldcg_u32(&a.alive[ap][i]) : 0u;
                        }
#pragma unroll
                        for (uint32_t r = 0; r < U; ++r) {
                            stv[r] = keep[r] ? ldcg_u32(&a.state[e[r]]) : 0u;
                            sv[r] = keep[r] ? ldcg_ll(&a.sup[e[r]]) : 0ll;
                        }
                        uint32_t n = 0, at[U];
#pragma unroll
                        for (uint32_t r = 0; r < U; ++r) {
                            keep[r] = keep[r] && stv[r] == kAlive;
                            if (keep[r]) {
                                a.snap[e[r]] = (int)sv[r];
                                const uint64_t d = a.inc_off[e[r] + 1] - a.inc_off[e[r]];
                                atomicAdd(&s_hist[bin_of((unsigned long long)sv[r])], 1u + (uint32_t)(d >> a.wshift));
                            }
                            const unsigned int mask = __ballot_sync(kFull, keep[r]);
                            at[r] = n + __popc(mask & ((1u << lane) - 1u));
                            n += __popc(mask);
                        }
                        if (anew && n) {
                            uint32_t base = 0;
                            if (lane == 0) base = atomicAdd(&ctl->n_alive[ap ^ 1u], n);
                            base = __shfl_sync(kFull, base, 0);
#pragma unroll
                            for (uint32_t r = 0; r < U; ++r)
                                if (keep[r]) a.alive[ap ^ 1u][base + at[r]] = e[r];
                        }
                    }
                    __syncthreads();
                    for (uint32_t i = threadIdx.x; i < kBins; i += kT)
                        if (s_hist[i]) atomicAdd(&ctl->hist[hno & 1u][i], s_hist[i]);
                    {
                        const Snap sn{{nullptr, nullptr, nullptr, nullptr, nullptr}, nullptr};
                        if (!grid_barrier(a, bar_no, sn, &s_v)) break;
                    }
                    if (anew) {
                        v_alive = (uint32_t)remaining;
                        ap ^= 1u;
                        if (gtid == 0) ctl->n_alive[ap ^ 1u] = 0;
                    }
                    // every block finds the class up to which the edges of the next
                    // part reach
                    constexpr uint32_t kPer = (kBins + kT - 1) / kT;
                    uint32_t mine[kPer], sum = 0;
#pragma unroll
                    for (uint32_t r = 0; r < kPer; ++r) {
                        const uint32_t b = threadIdx.x * kPer + r;
                        mine[r] = b < kBins ? __ldcg(&ctl->hist[hno & 1u][b]) : 0u;
                        sum += mine[r];
                    }
                    uint32_t total;
                    uint32_t cum = dev::block_excl_scan<uint32_t>(sum, &total);
                    if (hno == 0) {
                        // the largest weight within a factor of 8 in support
                        uint32_t run = cum, most = 0;
                        if (threadIdx.x == 0) s_cum = 0;
#pragma unroll
                        for (uint32_t r = 0; r < kPer; ++r) {
                            const uint32_t b = threadIdx.x * kPer + r;
                            run += mine[r];
                            if (b < kBins) s_hist[b] = run;
                        }
                        __syncthreads();
                        run = cum;
#pragma unroll
                        for (uint32_t r = 0; r < kPer; ++r) {
                            const uint32_t b = threadIdx.x * kPer + r;
                            if (b < kBins && mine[r]) {
                                const uint32_t w = s_hist[bin_of(8ull * (unsigned long long)bin_top(b))] - run;
                                most = w > most ? w : most;
                            }
                            run += mine[r];
                        }
                        if (most) atomicMax(&s_cum, most);
                        __syncthreads();
                        const uint32_t rest = total - s_hist[kLow];
                        narrow = (float)s_cum >= kNarrow * (float)total || (rest <= kRest && rest <= total / 20u);
                        if (narrow) break;
                        __syncthreads();  // (s_cum is used again)
                    }
                    if (!within) {
                        L.label = pno;
                        // (edges without butterflies still weigh in the first range, so that
                        // the ranges do not depend on how they are taken out)
                        const uint32_t gone = pno == first_free && n_zero < a.target ? n_zero : 0u;
                        total += gone;
                        if (pno + 1u >= a.max_parts || total <= a.target + a.target / 2u) {
                            // the rest is the last part: nothing is left to be told apart
                            for (uint32_t i = gtid; i < v_alive; i += nthreads) {
                                const uint32_t e = ldcg_u32(&a.alive[ap][i]);
                                if (ldcg_u32(&a.state[e]) == kAlive) a.phi[e] = pno;
                            }
                            ++pno;
                            break;
                        }
                        // the peel takes more edges than the class holds: the target
                        // is scaled by what the last part grew by
                        if (pno > first_free) {
                            const float grew = (float)(total_jump - total) / (float)picked;
                            aim = fminf(fmaxf((float)a.target / grew, (float)a.target / 32.f), (float)a.target);
                        }
                        const uint32_t want = aim < 1.f + (float)gone ? 1u : (uint32_t)aim - gone;
#pragma unroll
                        for (uint32_t r = 0; r < kPer; ++r) {
                            // the first class with a weight of at least `want` up to it
                            if (cum < want && cum + mine[r] >= want) {
                                s_bin = threadIdx.x * kPer + r;
                                s_cum = cum + mine[r];
                            }
                            cum += mine[r];
                        }
                        __syncthreads();
                        L.k = lim = bin_top(s_bin);
                        picked = s_cum + gone;
                        total_jump = total;
                        ++pno;
                    }
                    for (uint32_t i = gtid; i < kBins; i += nthreads) ctl->hist[(hno & 1u) ^ 1u][i] = 0;
                    ++hno;
                }
                // C2: their links become incidence items of this round
                uint32_t sel = 0;
                for (uint32_t i0 = gwarp * 32u * U; i0 < v_alive; i0 += nthreads * U) {
                    uint32_t e[U], stv[U], nseg[U], all = 0;
                    long long sv[U];
                    uint64_t ib[U], ie[U];
                    bool in[U];
#pragma unroll
                    for (uint32_t r = 0; r < U; ++r) {
                        const uint32_t i = i0 + 32u * r + lane;
                        in[r] = i < v_alive;
                        e[r] = in[r] ? ldcg_u32(&a.alive[ap][i]) : 0u;
                    }
#pragma unroll
                    for (uint32_t r = 0; r < U; ++r) {
                        stv[r] = in[r] ? ldcg_u32(&a.state[e[r]]) : 0u;
                        sv[r] = in[r] ? ldcg_ll(&a.sup[e[r]]) : 0ll;
                    }
#pragma unroll
                    for (uint32_t r = 0; r < U; ++r) {
                        in[r] = in[r] && stv[r] == kAlive && sv[r] <= lim;
                        ib[r] = in[r] ? a.inc_off[e[r]] : 0ull;
                        ie[r] = in[r] ? a.inc_off[e[r] + 1] : 0ull;
                    }
#pragma unroll
                    for (uint32_t r = 0; r < U; ++r) {
                        if (in[r]) {
                            join_batch(a, e[r], round, L);
                            ++sel;
                        }
                        nseg[r] = (uint32_t)((ie[r] - ib[r] + kSeg - 1) / kSeg);
                        all += nseg[r];
                    }
                    const uint32_t incl = dev::warp_incl_scan(all);
                    const uint32_t sum = __shfl_sync(kFull, incl, 31);
                    if (sum) {
                        uint32_t base = 0;
                        if (lane == 31) base = atomicAdd(&ctl->n_items[par], sum);
                        uint32_t slot = __shfl_sync(kFull, base, 31) + incl - all;
#pragma unroll
                        for (uint32_t r = 0; r < U; ++r)
                            for (uint32_t s2 = 0; s2 < nseg[r]; ++s2, ++slot) {
                                const uint64_t j = ib[r] + (uint64_t)s2 * kSeg;
                                const uint64_t left = ie[r] - j;
                                const uint32_t cnt = (uint32_t)(left < kSeg ? left : kSeg);
                                a.items[par][slot] =
                                    make_uint4(e[r], (uint32_t)j, (uint32_t)(j >> 32), cnt | (s2 == 0 ? 0x80000000u : 0u));
                            }
                    }
                }
                sel = dev::warp_sum(sel);
                if (lane == 0 && sel) atomicAdd(&ctl->n_edges[c3], sel);
                {
                    const Snap sn{{&ctl->n_edges[c3], &ctl->n_items[par], &ctl->n_bseg[b4], &ctl->n_bseg[bp], nullptr},
                                  nullptr};
                    if (!grid_barrier(a, bar_no, sn, &s_v)) break;
                }
                n_batch = s_v.u[0];
                n_items = s_v.u[1];
                nb_cur = s_v.u[2];
                nb_prev = s_v.u[3];
                if (gtid == 0) ctl->minsup = ~0ull;
            }
        } else if (level_jump) {
            if (gtid == 0) atomicAdd(&ctl->scanned, (unsigned long long)v_near);
            // L1: minimum over the near window, compacting it
            {
                unsigned long long best = ~0ull;
                for (uint32_t i0 = blockIdx.x * blockDim.x; i0 < v_near; i0 += nthreads) {
                    const uint32_t i = i0 + threadIdx.x;
                    bool keep = false;
                    uint32_t e = 0;
                    if (i < v_near) {
                        e = ldcg_u32(&a.near[L.nq][i]);
                        // state and support requested together
                        const uint32_t stv = ldcg_u32(&a.state[e]);
                        const unsigned long long sv = (unsigned long long)ldcg_ll(&a.sup[e]);
                        if (stv == kAlive) {
                            keep = true;
                            best = sv < best ? sv : best;
                        }
                    }
                    const unsigned int mask = __ballot_sync(kFull, keep);
                    if (mask) {
                        unsigned int base = 0;
                        if (lane == 0) base = atomicAdd(&ctl->n_near[L.nq ^ 1u], (unsigned)__popc(mask));
                        base = __shfl_sync(kFull, base, 0);
                        if (keep) a.near[L.nq ^ 1u][base + __popc(mask & ((1u << lane) - 1u))] = e;
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long y = __shfl_xor_sync(kFull, best, o);
                    best = y < best ? y : best;
                }
                if (lane == 0 && best != ~0ull) atomicMin(&ctl->minsup, best);
            }
            {
                const Snap sn{{nullptr, nullptr, nullptr, nullptr, &ctl->n_near[L.nq ^ 1u]}, &ctl->minsup};
                if (!grid_barrier(a, bar_no, sn, &s_v)) break;
            }
            unsigned long long mn = s_v.w;
            v_near = s_v.u[4];
            L.nq ^= 1u;
            if (gtid == 0) ctl->n_near[L.nq ^ 1u] = 0;
            if (mn == ~0ull) {
                // the window holds no alive edge: rebuild it from all alive edges.
                // W1: overall minimum, compacting the alive list
                if (gtid == 0) atomicAdd(&ctl->scanned, (unsigned long long)v_alive);
                unsigned long long best = ~0ull;
                for (uint32_t i0 = blockIdx.x * blockDim.x; i0 < v_alive; i0 += nthreads) {
                    const uint32_t i = i0 + threadIdx.x;
                    bool keep = false;
                    uint32_t e = 0;
                    if (i < v_alive) {
                        e = ldcg_u32(&a.alive[ap][i]);
                        const uint32_t stv = ldcg_u32(&a.state[e]);
                        const unsigned long long sv = (unsigned long long)ldcg_ll(&a.sup[e]);
                        if (stv == kAlive) {
                            keep = true;
                            best = sv < best ? sv : best;
                        }
                    }
                    const unsigned int mask = __ballot_sync(kFull, keep);
                    if (mask) {
                        unsigned int base = 0;
                        if (lane == 0) base = atomicAdd(&ctl->n_alive[ap ^ 1u], (unsigned)__popc(mask));
                        base = __shfl_sync(kFull, base, 0);
                        if (keep) a.alive[ap ^ 1u][base + __popc(mask & ((1u << lane) - 1u))] = e;
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const unsigned long long y = __shfl_xor_sync(kFull, best, o);
                    best = y < best ? y : best;
                }
                if (lane == 0 && best != ~0ull) atomicMin(&ctl->minsup2, best);
                {
                    const Snap sn{{nullptr, nullptr, nullptr, nullptr, &ctl->n_alive[ap ^ 1u]}, &ctl->minsup2};
                    if (!grid_barrier(a, bar_no, sn, &s_v)) break;
                }
                mn = s_v.w;
                if (mn == ~0ull) break;  // no alive edge: cannot happen while remaining > 0
                v_alive = s_v.u[4];
                L.khi = window_top((long long)mn);
                ap ^= 1u;
                if (gtid == 0) ctl->n_alive[ap ^ 1u] = 0;
                // W2: list every alive edge below the new window top (one
                // counter atomic per warp: the list can take most edges)
                if (gtid == 0) atomicAdd(&ctl->scanned, (unsigned long long)v_alive);
                for (uint32_t i0 = gwarp * 32u; i0 < v_alive; i0 += nthreads) {
                    const uint32_t i = i0 + lane;
                    uint32_t e = 0;
                    bool keep = false;
                    if (i < v_alive) {
                        e = ldcg_u32(&a.alive[ap][i]);
                        keep = ldcg_ll(&a.sup[e]) < L.khi;
                    }
                    const unsigned int mask = __ballot_sync(kFull, keep);
                    if (mask) {
                        unsigned int base = 0;
                        if (lane == 0) base = atomicAdd(&ctl->n_near[L.nq], (unsigned)__popc(mask));
                        base = __shfl_sync(kFull, base, 0);
                        if (keep) a.near[L.nq][base + __popc(mask & ((1u << lane) - 1u))] = e;
                    }
                }
                if (gtid == 0) atomicAdd(&ctl->windows, 1ull);
                {
                    const Snap sn{{nullptr, nullptr, nullptr, nullptr, &ctl->n_near[L.nq]}, nullptr};
                    if (!grid_barrier(a, bar_no, sn, &s_v)) break;
                }
                v_near = s_v.u[4];
                if (gtid == 0) ctl->minsup2 = ~0ull;
            }
            if ((long long)mn > L.k) L.k = (long long)mn;
            L.label = (uint32_t)L.k;
            if ((unsigned long long)L.k > 0xFFFFFFFFull) {
                if (gtid == 0) atomicOr(&ctl->err, kErrPeelOverflow);
                break;
            }
            // L2: the batch is every window edge with support <= k; their
            // links become incidence items of this round.  A large window
            // (a level can select millions of edges) takes its item slots
            // with one atomic per warp; a small one per edge, which is faster
            // when only a few edges are selected.
            uint32_t sel = 0;
            if (gtid == 0) atomicAdd(&ctl->scanned, (unsigned long long)v_near);
            if (v_near > kWarpSlotsMin) {
                for (uint32_t i0 = gwarp * 32u; i0 < v_near; i0 += nthreads) {
                    const uint32_t i = i0 + lane;
                    uint32_t e = 0, nseg = 0;
                    uint64_t ib = 0, ie = 0;
                    if (i < v_near) {
                        e = ldcg_u32(&a.near[L.nq][i]);
                        // state, support and link range requested together
                        const uint32_t stv = ldcg_u32(&a.state[e]);
                        const long long sv = ldcg_ll(&a.sup[e]);
                        const uint64_t b0 = a.inc_off[e], b1 = a.inc_off[e + 1];
                        if (stv == kAlive && sv <= L.k) {
                            join_batch(a, e, round, L);
                            ++sel;
                            ib = b0;
                            ie = b1;
                            nseg = (uint32_t)((ie - ib + kSeg - 1) / kSeg);
                        }
                    }
                    const uint32_t incl = dev::warp_incl_scan(nseg);
                    const uint32_t all = __shfl_sync(kFull, incl, 31);
                    if (all) {
                        uint32_t base = 0;
                        if (lane == 31) base = atomicAdd(&ctl->n_items[par], all);
                        uint32_t slot = __shfl_sync(kFull, base, 31) + incl - nseg;
                        for (uint32_t s2 = 0; s2 < nseg; ++s2, ++slot) {
                            const uint64_t j = ib + (uint64_t)s2 * kSeg;
                            const uint64_t left = ie - j;
                            const uint32_t cnt = (uint32_t)(left < kSeg ? left : kSeg);
                            a.items[par][slot] =
                                make_uint4(e, (uint32_t)j, (uint32_t)(j >> 32), cnt | (s2 == 0 ? 0x80000000u : 0u));
                        }
                    }
                }
            } else {
                for (uint32_t i = gtid; i < v_near; i += nthreads) {
                    const uint32_t e = ldcg_u32(&a.near[L.nq][i]);
                    const uint32_t stv = ldcg_u32(&a.state[e]);
                    const long long sv = ldcg_ll(&a.sup[e]);
                    const uint64_t b0 = a.inc_off[e], b1 = a.inc_off[e + 1];
                    if (stv == kAlive && sv <= L.k) {
                        join_batch(a, e, round, L);
                        push_items<kSeg>(a, e, par, b0, b1);
                        ++sel;
                    }
                }
            }
            sel = dev::warp_sum(sel);
            if (lane == 0 && sel) atomicAdd(&ctl->n_edges[c3], sel);
            if (gtid == 0) atomicAdd(&ctl->levels, 1ull);
            {
                const Snap sn{{&ctl->n_edges[c3], &ctl->n_items[par], &ctl->n_bseg[b4], &ctl->n_bseg[bp],
                               &ctl->n_near[L.nq]},
                              nullptr};
                if (!grid_barrier(a, bar_no, sn, &s_v)) break;
            }
            n_batch = s_v.u[0];
            n_items = s_v.u[1];
            nb_cur = s_v.u[2];
            nb_prev = s_v.u[3];
            v_near = s_v.u[4];
            if (gtid == 0) ctl->minsup = ~0ull;
        }

        if (gtid == 0) {
            ctl->n_edges[(round + 2u) % 3u] = 0;  // batch of round - 1: read before the last barrier
            ctl->n_bseg[(round + 2u) & 3u] = 0;   // bloom items of round - 2: C cleared in round - 1
        }

        // ---------------- incidence phase (only for queued link lists)
        if (n_items > 0) {
            if (gtid == 0) atomicAdd(&ctl->inc_phases, 1ull);
            constexpr uint32_t U = 4;  // links a lane has in flight
            Slots t;
            const bool stock = n_items > nwarps;  // a small phase takes its places one atomic a warp
            for (uint32_t base = gwarp; base < n_items; base += nwarps * 32u) {
                const uint32_t i = base + lane * nwarps;
                const uint4 it = i < n_items ? __ldcg(&a.items[par][i]) : make_uint4(0, 0, 0, 0);
                const uint32_t cnt = it.w & 0x7FFFFFFFu;
                // the links of the warp's items side by side (as in the bloom phase)
                const uint32_t incl = dev::warp_incl_scan(cnt);
                const uint32_t all = __shfl_sync(kFull, incl, 31);
                const uint64_t start = ((uint64_t)it.z << 32 | it.y) + cnt - incl;
                for (uint32_t x0 = 0; x0 < all; x0 += 32u * U) {
                    uint2 l[U];
                    uint32_t B[U];
                    bool won[U];
#pragma unroll
                    for (uint32_t r = 0; r < U; ++r) {
                        const uint32_t x = x0 + lane + 32u * r;
                        uint32_t j = 0;  // the item of link x: the first with incl > x
#pragma unroll
                        for (uint32_t step = 16; step > 0; step >>= 1)
                            if (__shfl_sync(kFull, incl, j + step - 1u) <= x) j += step;
                        const uint64_t at = __shfl_sync(kFull, start, j) + x;
                        won[r] = x < all;
                        l[r] = won[r] ? a.inc[at] : make_uint2(0u, 0u);
                        B[r] = l[r].y & 0x7FFFFFFFu;
                    }
                    // the first edge of the batch to stamp a pair kills it (once)
                    kill_pairs<U>(a, l, won, round);
                    if (stock) warp_kills<kSeg, U, 2>(a, round, B, won, lane, t);
                    else warp_kills<kSeg, U, 0>(a, round, B, won, lane, t);
                }
            }
            fill_empty(a, b4, t, lane);
            {
                const Snap sn{{nullptr, nullptr, &ctl->n_bseg[b4], nullptr, nullptr}, nullptr};
                if (!grid_barrier(a, bar_no, sn, &s_v)) break;
            }
            nb_cur = s_v.u[2];
        }

        // ---------------- bloom phase of this round, kills of the next
        if (gtid == 0) ctl->n_items[par] = 0;
        {
            const uint32_t q = round + 1u;
            for (uint32_t base = gwarp; base < nb_cur; base += nwarps * 32u) {
                const uint32_t i = base + lane * nwarps;
                const uint4 it = i < nb_cur ? __ldcg(&a.bseg[b4][i]) : make_uint4(0, 0, 0, 0);
                const uint32_t cnt = it.z & 0x7FFFFFFFu;
                // the bloom's kills of this round, and its number at round start:
                // recorded after the last round that touched it, or by its head
                // item in this round already
                uint32_t c = 0, k0 = 0;
                if (cnt) {
                    BloomWord *b = a.blooms + it.x;
                    const unsigned long long w = __ldcg(&b->bw);
                    c = __ldcg(&b->C[c3]);
                    k0 = (uint32_t)w + ((uint32_t)(w >> 32) == round ? c : 0u);
                    if (it.z >> 31) b->bw = (unsigned long long)round << 32 | (uint32_t)(k0 - c);
                }
                slots += cnt;
                // the warp's items side by side: lane l takes slots l, l + 32, ...
                // of their concatenation, so small items fill the warp too
                const uint32_t incl = dev::warp_incl_scan(cnt);
                const uint32_t all = __shfl_sync(kFull, incl, 31);
                constexpr uint32_t U = R < 2u ? 2u : R;  // slots a lane has in flight
                for (uint32_t x0 = 0; x0 < all; x0 += 32u * U) {
                    uint32_t d[U], kB[U], cc[U];
                    uint2 pr[U];
#pragma unroll
                    for (uint32_t r = 0; r < U; ++r) {
                        const uint32_t x = x0 + lane + 32u * r;
                        uint32_t j = 0;  // the item of slot x: the first with incl > x
#pragma unroll
                        for (uint32_t step = 16; step > 0; step >>= 1)
                            if (__shfl_sync(kFull, incl, j + step - 1u) <= x) j += step;
                        const bool act = x < all;
                        const uint32_t p = __shfl_sync(kFull, it.y + cnt - incl, j) + x;
                        kB[r] = __shfl_sync(kFull, k0, j);
                        cc[r] = __shfl_sync(kFull, c, j);
                        d[r] = act ? __ldcg(&a.died[p]) : (round + 2u) << 2;  // inactive: no case applies
                        pr[r] = act ? a.pairs[p] : make_uint2(0, 0);
                    }
                    apply_slots<kSeg, U>(a, d, pr, cc, kB, L, round, upd, s_je, &s_jn);
                }
            }
            // clear C of the blooms the previous round touched (threads from
            // the top of the grid, away from the bloom items above)
            const uint32_t cp = (round + 2u) % 3u;
            for (uint32_t i = nthreads - 1u - gtid; i < nb_prev; i += nthreads) {
                const uint4 it = __ldcg(&a.bseg[bp][i]);
                if (it.z >> 31) a.blooms[it.x].C[cp] = 0;
            }

            // the block kills the twin pairs of the edges it listed
            __syncthreads();
            const uint32_t njr = s_jn;
            const uint32_t nj = njr < a.join_cap ? njr : a.join_cap;
            if (nj > 0) {
                uint32_t e = 0, d = 0;
                uint64_t ib = 0;
                if (threadIdx.x < nj) {
                    e = s_je[threadIdx.x];
                    join_batch(a, e, q, L);
                    ib = a.inc_off[e];
                    const uint64_t dl = a.inc_off[e + 1] - ib;
                    d = dl > a.block_links ? a.block_links + 1u : (uint32_t)dl;  // longer lists are queued
                }
                uint32_t total = 0;
                const uint32_t off = dev::block_excl_scan<uint32_t>(d, &total);
                if (threadIdx.x < nj) {
                    s_joff[threadIdx.x] = off;
                    s_jd[threadIdx.x] = d;
                    s_jib[threadIdx.x] = ib;
                    if (off + d > a.block_links) push_items<kSeg>(a, e, q & 1u, ib, a.inc_off[e + 1]);
                }
                if (threadIdx.x == 0) atomicAdd(&ctl->n_edges[q % 3u], nj);
                __syncthreads();
                const uint32_t lim = total < a.block_links ? total : a.block_links;
                uint2 l[2];
                uint32_t B[2];
                bool won[2];
#pragma unroll
                for (uint32_t r = 0; r < 2; ++r) {
                    const uint32_t x = threadIdx.x + r * kT;
                    won[r] = false;
                    l[r] = make_uint2(0u, 0u);
                    if (x < lim) {
                        const uint32_t j = dev::last_le_u32(s_joff, nj, x);
                        if (s_joff[j] + s_jd[j] <= a.block_links) {
                            won[r] = true;
                            l[r] = a.inc[s_jib[j] + (x - s_joff[j])];
                        }
                    }
                    B[r] = l[r].y & 0x7FFFFFFFu;
                }
                // the first edge of the batch to stamp a pair kills it (once)
                kill_pairs<2>(a, l, won, q);
                Slots none;
                if (kCoarse && lim > kT / 2u) warp_kills<kSeg, 2, 1>(a, q, B, won, lane, none);
                else warp_kills<kSeg, 2, 0>(a, q, B, won, lane, none);
                if (threadIdx.x == 0) s_jn = 0;
            }
        }
        {
            // next round: its batch, incidence items, bloom items, this
            // round's bloom items (C to clear) and the near list size
            const uint32_t q = round + 1u;
            const Snap sn{{&ctl->n_edges[q % 3u], &ctl->n_items[q & 1u], &ctl->n_bseg[q & 3u], &ctl->n_bseg[b4],
                           &ctl->n_near[L.nq]},
                          nullptr};
            if (!grid_barrier(a, bar_no, sn, &s_v)) break;
        }
        remaining -= n_batch;
        ++round;
        n_batch = s_v.u[0];
        n_items = s_v.u[1];
        nb_cur = s_v.u[2];
        nb_prev = s_v.u[3];
        v_near = s_v.u[4];
        level_jump = remaining > 0 && n_batch == 0;
    }
    upd = dev::warp_sum(upd);
    if (lane == 0 && upd) atomicAdd(in_first ? &ctl->first_updates : &ctl->updates, upd);
    slots = dev::warp_sum(slots);
    if (lane == 0 && slots) atomicAdd(&ctl->slots, slots);
    if (gtid == 0 && in_first) ctl->first_rounds = round;
    if (gtid == 0) {
        ctl->rounds = round;
        ctl->kfinal = (unsigned long long)L.k;
        ctl->n_parts = pno;
        ctl->narrow = narrow;
    }
}

// Edges already assigned (mask set) start in the permanent state: never alive,
// never queued.  So do, for a coarse peel from level 0 (zero_part not null), the
// edges in no butterfly: they are the batch of level 0 and change nothing else.
constexpr uint32_t kPerm = 0xFFFFFFFEu;
__global__ void k_peel_init(const uint64_t *support, uint64_t m, int *sup, uint32_t *state,
                            const uint8_t *assigned, uint32_t *alive, uint32_t *zero_part, unsigned int *n_zero) {
    uint32_t zeros = 0;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m;
         i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t v = support[i];
        const bool fixed = assigned && assigned[i], zero = !fixed && zero_part && v == 0;
        sup[i] = (int)v;
        state[i] = fixed || zero ? kPerm : kAlive;
        alive[i] = (uint32_t)i;
        if (zero) {
            zero_part[i] = 0;
            ++zeros;
        }
    }
    zeros = dev::warp_sum(zeros);
    if ((threadIdx.x & 31) == 0 && zeros) atomicAdd(n_zero, zeros);
}

// Bloom words: no round has touched the bloom yet, k_B from the index.
__global__ void k_bloom_words(const uint32_t *bloom_k, uint64_t nb, BloomWord *blooms) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < nb;
         i += (uint64_t)gridDim.x * blockDim.x) {
        uint4 *w = reinterpret_cast<uint4 *>(blooms + i);
        w[0] = make_uint4(bloom_k[i], 0xFFFFFFFFu, 0u, 0u);
        w[1] = make_uint4(0u, 0u, 0u, 0u);
    }
}

inline unsigned grid_for(uint64_t items, int threads, unsigned cap) {
    uint64_t g = (items + threads - 1) / threads;
    if (g == 0) g = 1;
    return (unsigned)(g < cap ? g : cap);
}

}  // namespace

cudaError_t peel(const Index &ix, const uint64_t *support, uint32_t *phi_out, PeelResult &res,
                 int num_sms, Alloc &al, int seg, const PeelOpts *opts) {
    const bool coarse = opts && opts->snap;
    // (a coarse peel has no kernel of 64-entry items: every size below goes by the
    // items of the kernel that is launched)
    const uint32_t kSeg = seg == 128 ? 128u : seg == 64 && !coarse ? 64u : 32u;
    const uint32_t kT = (uint32_t)peel_threads(kSeg);
    const uint32_t kJoinCap = kT, kBlockLinks = 2 * kT;
    const uint64_t m = ix.m;
    res = PeelResult{};
    if (m == 0 || (opts && opts->assigned && opts->m_active == 0)) return cudaSuccess;
    int bps = 0;
    void *kfn = coarse ? (kSeg == 128 ? (void *)k_peel<128, true> : (void *)k_peel<32, true>)
                       : kSeg == 128 ? (void *)k_peel<128, false>
                                     : kSeg == 64 ? (void *)k_peel<64, false> : (void *)k_peel<32, false>;
    BT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kfn, (int)kT, 0));
    if (bps < 1) return cudaErrorCooperativeLaunchTooLarge;
    const dim3 grid((unsigned)(num_sms * bps)), block(kT);
    // one round queues each edge and each bloom at most once
    const uint64_t item_cap = m + (2 * ix.w2) / kSeg + 2;
    // (beside the places a warp has taken and not filled)
    const uint64_t bseg_cap = ix.nb + ix.w2 / kSeg + (uint64_t)grid.x * (kT / 32) * kTake + 2;
    PeelArgs a{};
    a.m = m;
    a.inc_off = ix.inc_off;
    a.inc = ix.inc;
    a.pairs = ix.pairs;
    a.phi = phi_out;
    a.sup = al.get<int>(m);
    a.state = al.get<uint32_t>(m);
    a.died = al.get<uint32_t>(ix.w2);
    a.bloom_off = ix.bloom_off;
    a.blooms = al.get<BloomWord>(ix.nb);
    for (int i = 0; i < 4; ++i) a.bseg[i] = al.get<uint4>(bseg_cap);
    for (int i = 0; i < 2; ++i) {
        a.items[i] = al.get<uint4>(item_cap);
        a.alive[i] = al.get<uint32_t>(m);
        a.near[i] = al.get<uint32_t>(m);
    }
    a.item_cap = item_cap;
    a.bseg_cap = bseg_cap;
    a.ctl = al.get<Ctl>(1);
    {
        const bt_limits *lim = al.limits;
        uint64_t rl = m + 1 < kMaxRounds ? m + 1 : kMaxRounds;
        if (lim && lim->peel_round_limit && lim->peel_round_limit < rl) rl = lim->peel_round_limit;
        a.round_limit = rl;
        a.barrier_timeout_ns = (lim && lim->barrier_timeout_ns) ? lim->barrier_timeout_ns : kBarrierTimeoutNs;
        a.hold_barrier = lim ? lim->hold_barrier : 0;
        a.join_cap = (lim && lim->join_cap && lim->join_cap < kJoinCap) ? lim->join_cap : kJoinCap;
        a.block_links = (lim && lim->block_links && lim->block_links < kBlockLinks) ? lim->block_links : kBlockLinks;
    }
    a.m_active = (opts && opts->assigned) ? opts->m_active : m;
    a.k_init = opts ? opts->k_init : 0;
    a.assign_from = opts ? opts->assign_from : 0;
    a.snap = coarse ? opts->snap : nullptr;
    if (coarse) {
        // weights add up to less than 2^31
        while ((ix.links >> a.wshift) >> 30) ++a.wshift;
        const uint64_t all = m + (ix.links >> a.wshift), t = all / (opts->parts_hint ? opts->parts_hint : 1);
        a.target = (uint32_t)(t ? t : 1);
    }
    a.max_parts = coarse ? opts->max_parts : 0;
    if (al.err != cudaSuccess) return al.err;
    cudaStream_t st = al.stream;
    Ctl h{};
    h.n_alive[0] = (unsigned int)m;
    h.minsup = ~0ull;
    h.minsup2 = ~0ull;
    BT_CUDA(cudaMemsetAsync(a.ctl, 0, sizeof(Ctl), st));
    BT_CUDA(cudaMemcpyAsync(a.ctl, &h, offsetof(Ctl, hist), cudaMemcpyHostToDevice, st));
    k_peel_init<<<grid_for(m, 256, (unsigned)num_sms * 16), 256, 0, st>>>(
        support, m, a.sup, a.state, opts ? opts->assigned : nullptr, a.alive[0],
        coarse && a.k_init == 0 ? a.phi : nullptr, &a.ctl->n_zero);
    al.launches++;
    BT_CUDA(cudaMemsetAsync(a.died, 0xFF, sizeof(uint32_t) * (ix.w2 ? ix.w2 : 1), st));
    if (ix.nb) {
        k_bloom_words<<<grid_for(ix.nb, 256, (unsigned)num_sms * 16), 256, 0, st>>>(ix.bloom_k, ix.nb, a.blooms);
        al.launches++;
    }
    void *kargs[] = {&a};
    BT_CUDA(cudaLaunchCooperativeKernel(kfn, grid, block, kargs, 0, st));
    al.launches++;
    BT_CUDA(cudaMemcpyAsync(&h, a.ctl, offsetof(Ctl, hist), cudaMemcpyDeviceToHost, st));
    BT_CUDA(cudaStreamSynchronize(st));
    if (h.err & kErrBarrier) res.status = BT_ERR_CUDA;
    else if (h.err & kErrPeelOverflow) res.status = BT_ERR_OVERFLOW;
    else if (h.err & kErrRounds) res.status = BT_ERR_NOCONVERGE;
    res.rounds = h.rounds;
    res.levels = h.levels;
    res.windows = h.windows;
    res.updates = h.updates;
    res.slots = h.slots;
    res.scanned = h.scanned;
    res.kmax = h.kfinal;
    res.inc_phases = h.inc_phases;
    res.parts = h.n_parts;
    res.narrow = h.narrow != 0;
    res.zero_edges = h.n_zero;
    res.first_rounds = h.first_rounds;
    res.first_levels = h.first_levels;
    res.first_updates = h.first_updates;
    al.put(a.sup);
    al.put(a.state);
    al.put(a.died);
    al.put(a.blooms);
    for (int i = 0; i < 4; ++i) al.put(a.bseg[i]);
    for (int i = 0; i < 2; ++i) {
        al.put(a.items[i]);
        al.put(a.alive[i]);
        al.put(a.near[i]);
    }
    al.put(a.ctl);
    return cudaSuccess;
}

}  // namespace bt
