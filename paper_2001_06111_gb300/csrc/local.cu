// Peeling by independent parts, one thread block a part (Section V-B, Alg. 5).
//
// A part holds the edges whose bitruss numbers lie in one range (split.cu), with
// their supports when all lower parts are gone; removals in higher parts come
// later and change nothing here.  So the batches S of Alg. 5 inside the range
// depend on this part alone: a block peels the whole part by itself, all parts at
// once, and the phases of a round are separated by block barriers instead of
// the grid barriers of peel.cu.  The batches, and with them rounds, levels and
// support updates, are those of the one peel of the whole graph (an update of an
// edge of a higher part is counted where Alg. 5 makes it and left out).  On the
// 2M-edge graph 39,928 rounds of about 10 us became at most 3,000 a part, of
// 6-15 us, in 85 parts side by side: the peel went from 384 to 69 ms (39 of them
// the coarse peel, 10 the split, 20 this kernel); with planted bicliques (2.4M
// edges) from 484 to 112 ms; 20,000 edges from 7.8 to 2.0 ms; a batch of 384
// graphs from 209 to 82 ms.
//
// One round (batch S of edges with support <= k, bloom numbers k_B):
//   phase 1, over the links of S: a pair of bloom B dies when its other edge is
//     still there (or is in S too and has the larger id, so that a pair counts
//     once); C(B) += 1, and the other edge, if outside S, loses k_B - 1
//     (Lemma 2).  A pair is dead exactly when one of its edges is, so no death
//     stamp is kept: links carry the twin edge itself.
//   phase 2, over the blooms with C(B) > 0: both edges of every pair still
//     alive lose C(B), then k_B -= C(B).
// An edge joins the next batch when one decrement carries its support from
// above k to <= k.  When a batch ends empty, k jumps to the minimum support of
// a window of low supports, which is rebuilt from the alive edges when it
// runs out (as in peel.cu).
//
// What bounds it: the chain of dependent accesses of a round and, in heavy
// rounds, the number of accesses one SM keeps in flight.  So
//   * links and pairs are laid side by side by a block scan over the batch's
//     edges (the touched blooms) and dealt out one a thread, kU a turn;
//   * the supports of a part of up to kCap edges, the lists of touched blooms
//     and the next batch's link ranges stay in shared memory: a round waits
//     for the links, the bloom counters, the bloom records and the pairs;
//   * k_B and C(B) of a bloom are one 64-bit word, so a kill is one atomic and no
//     load: a load beside an atomic on the same sector cost 14 instead of 5 ns
//     a link an SM with all SMs busy;
//   * a bloom's record and up to two of its pairs share one 32-byte sector;
//   * a part with more than four times the mean links, or too many edges for a
//     block's shared memory, is peeled by a cluster of 16 blocks (a dense
//     biclique of 77,000 edges: 17 rounds, 290 ms by one block).  1,024 threads
//     leave 64 registers a thread, of which the cluster's kernel spills 36 bytes.
//
// Supports are below m < 2^31 (k butterflies on an edge need k other edges, one
// opposite edge each), so they are kept as 32-bit integers here.
#include <limits.h>

#include <cooperative_groups.h>

#include "bt_device.cuh"
#include "bt_internal.cuh"

namespace cg = cooperative_groups;

namespace bt {
namespace {

// threads a block: with 512 the peel of the 2M-edge graph took 73.3 instead of
// 69.0 ms, of planted bicliques 131 instead of 118, of 1,003 edges 0.69 instead
// of 0.74
constexpr int kNT = 1024;
constexpr unsigned kAll = 0xffffffffu;
constexpr uint32_t kCluster = 16;  // blocks of the cluster that peels a heavy part
constexpr uint32_t kU = 4;         // links or pairs a thread has in flight
constexpr uint32_t kTouch = 4096;  // touched blooms a block lists in shared memory
constexpr uint32_t kFront = 512;   // edges of a batch whose link ranges are kept there
constexpr uint32_t kCap = kBlockEdges;  // edges of a part whose supports are kept there
// supports of a part in shared memory also tell the state: an edge of the
// batch, an edge of an earlier batch, or (not negative) one still there
constexpr int kBatch = INT_MIN, kDead = INT_MIN + 1;

struct LocalArgs {
    const uint32_t *part_e, *part_b;  // [np + 1] first edge / bloom slot of each part
    const uint32_t *order;            // parts, heaviest first
    uint32_t np;
    uint32_t *queue;
    const uint4 *er;    // per edge: first link, links, initial support
    const uint2 *inc;   // per edge: (twin | higher-part flag << 31, bloom)
    const uint2 *pairs;
    BloomRec *bl;
    int *sup;           // [m] supports and states of the parts that clusters peel
    uint32_t *st;
    uint32_t *fq;       // [m] batches of a part, one after another
    uint32_t *near[2];  // [m] window lists
    uint32_t *alive[2];
    uint32_t *touch;    // [nb] touched blooms beyond kTouch a block
    uint32_t *phi;
    uint32_t *depth;    // [m + 1] rounds of level k (the most any part needed)
    unsigned long long *stats;  // updates, pair slots, scanned entries
    uint32_t *err;
    uint64_t round_limit;
    long long assign_from;
    bool assigned;  // some twins are assigned edges: no update is counted for them
};

struct Shared {
    // kept by block 0 for the whole cluster
    uint32_t nj[2];        // edges that joined the next batch, by round parity
    uint32_t nover[2];     // touched blooms listed in a.touch
    uint32_t nn[2], na, sel;
    int mn, k, khi;        // a level jump's results
    uint32_t tail, cur;
    uint32_t part;
    // each block's own
    uint32_t nt[2];        // touched blooms listed here
    unsigned long long total64;
    uint32_t n;            // items laid side by side, their entries
    uint32_t off[kNT + 1]; // first entry of each
    uint32_t id[kNT + 1], c[kNT + 1];
    unsigned long long at[kNT + 1];  // entry x of item j is at address at[j] + 8 x
    uint32_t touch[kTouch];
    uint4 front[2][kFront];  // records of the first kFront edges of a batch
    uint32_t fe[2][kFront];  // and the edges, by round parity
};

static_assert(sizeof(Shared) + sizeof(int) * kCap <= 226 * 1024, "shared memory of a block");

template <typename T>
__device__ __forceinline__ T warp_min(T x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const T y = __shfl_xor_sync(kAll, x, o);
        x = y < x ? y : x;
    }
    return x;
}

__device__ __forceinline__ int window_top(int kmin) {
    const int w = kmin / 64;
    const long long t = (long long)kmin + (w < 8 ? 8 : w);
    return t > INT_MAX ? INT_MAX : (int)t;
}

// Lanes with `keep` set take consecutive places of a shared counter.
__device__ __forceinline__ uint32_t warp_place(uint32_t *ctr, bool keep, int lane) {
    const unsigned mask = __ballot_sync(kAll, keep);
    if (!mask) return 0;
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(ctr, (uint32_t)__popc(mask));
    return __shfl_sync(kAll, base, 0) + __popc(mask & ((1u << lane) - 1u));
}

__device__ __forceinline__ void copy_async(uint4 *to, const uint4 *from) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from)
                 : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The state of one part's peel.  kC: by the blocks of a cluster, with supports
// and states in global memory; else by one block (a part of up to kCap edges),
// with supports in shared memory.
template <bool kC>
struct Part {
    static constexpr bool kS = !kC;
    const LocalArgs &a;
    Shared &s;         // this block's
    Shared &s0;        // block 0's
    const uint32_t e0, b0, rank, nranks;
    int *sup;
    uint32_t *st;
    int k = -1, khi = INT_MIN;
    uint32_t round = 0, tail = 0, cur = 0;
    unsigned long long upd = 0, slots = 0;

    __device__ __forceinline__ void barrier() const {
        if constexpr (!kC) copies_done();
        if constexpr (kC) cg::this_cluster().sync();
        else __syncthreads();
    }
    // Whether edge e is still there, for a level jump: its support, or a
    // negative number.
    __device__ __forceinline__ int alive_sup(uint32_t e) const {
        if constexpr (kS) return sup[e];
        const int v = __ldcg(&sup[e]);
        return __ldcg(&st[e]) == kAlive ? v : -1;
    }
    // Edge t as the twin of a link of the batch: 0 gone, 1 in the batch, 2 there.
    __device__ __forceinline__ uint32_t twin_state(uint32_t t) const {
        if constexpr (kS) {
            const int v = sup[t];
            return v == kDead ? 0u : v == kBatch ? 1u : 2u;
        }
        const uint32_t v = __ldcg(&st[t]);
        return v < round ? 0u : v == round ? 1u : 2u;
    }
    // Whether edge e is there after the batch's removal (one that joined the
    // next batch still is).
    __device__ __forceinline__ bool remains(uint32_t e) const {
        if constexpr (kS) return sup[e] >= 0;
        return __ldcg(&st[e]) > round;
    }
    // Edge e joins, as number j, the batch that starts at place `base` of the queue.
    __device__ __forceinline__ void settle(uint32_t e, uint32_t stamp, uint32_t base, uint32_t j) {
        if constexpr (!kS) st[e] = stamp;
        if (k >= a.assign_from) a.phi[e0 + e] = (uint32_t)k;
        if (!kC && j < kFront) {
            // the link range follows by itself: no thread waits for it before
            // the phase ends
            s.fe[stamp & 1u][j] = e;
            copy_async(&s.front[stamp & 1u][j], a.er + e0 + e);
        } else {
            a.fq[e0 + base + j] = e;
        }
    }
    // Edges e[i] lose d[i] butterflies (none where d[i] is 0).  All decrements go
    // out before a result is looked at.
    template <uint32_t N>
    __device__ __forceinline__ void lose(const uint32_t (&e)[N], const int (&d)[N]) {
        int old[N];
#pragma unroll
        for (uint32_t i = 0; i < N; ++i) old[i] = d[i] ? atomicSub(&sup[e[i]], d[i]) : INT_MIN;
#pragma unroll
        for (uint32_t i = 0; i < N; ++i) {
            const int now = old[i] - d[i];
            if (now <= k) {
                if (old[i] > k) settle(e[i], round + 1u, tail, atomicAdd(&s0.nj[round & 1u], 1u));
            } else if (old[i] >= khi && now < khi) {
                a.near[cur][e0 + atomicAdd(&s0.nn[cur], 1u)] = e[i];
            }
        }
    }
    // Lays up to kNT items of len entries, one a thread, side by side, empty
    // ones left out: fills s.off, s.id, s.c and s.at.  Returns the entries.
    // Called by the whole block, `n` threads with an item.
    __device__ __forceinline__ unsigned long long lay(uint32_t n, uint32_t len, uint32_t id, uint32_t c,
                                                      const uint2 *at) {
        const uint32_t tid = threadIdx.x;
        uint32_t j, x;
        unsigned long long all;
        if (n <= 32u) {
            if (tid < 32u) {
                const unsigned has = __ballot_sync(kAll, len > 0u);
                const unsigned long long incl = dev::warp_incl_scan((unsigned long long)len);
                j = __popc(has & ((1u << tid) - 1u));
                if (len) {
                    s.off[j] = (uint32_t)incl - len;
                    s.id[j] = id;
                    s.c[j] = c;
                    s.at[j] = (unsigned long long)at - 8ull * (incl - len);
                }
                if (tid == 31u) {
                    s.n = __popc(has);
                    s.off[__popc(has)] = (uint32_t)incl;
                    s.total64 = incl;
                }
            }
            __syncthreads();
            return s.total64;
        }
        const unsigned long long ex =
            dev::block_excl_scan<unsigned long long>((unsigned long long)(len > 0u) << 48 | len, &all);
        j = (uint32_t)(ex >> 48);
        x = (uint32_t)ex;
        if (len) {
            s.off[j] = x;
            s.id[j] = id;
            s.c[j] = c;
            s.at[j] = (unsigned long long)at - 8ull * x;
        }
        all &= (1ull << 48) - 1ull;
        if (tid == kNT - 1u) {
            const uint32_t cnt = j + (len > 0u);
            s.n = cnt;
            s.off[cnt] = (uint32_t)all;
        }
        __syncthreads();
        return all;
    }
    __device__ __forceinline__ const uint2 *entry(uint32_t j, uint32_t x) const {
        return reinterpret_cast<const uint2 *>(s.at[j] + 8ull * x);
    }
    // The batch's edges in shared memory receive state v.
    __device__ __forceinline__ void mark(uint32_t head, uint32_t F, int v) {
        for (uint32_t i = threadIdx.x; i < F; i += kNT)
            sup[i < kFront ? s.fe[round & 1u][i] : __ldcg(&a.fq[e0 + head + i])] = v;
    }

    // Entries [w, w + 32 U) of the batch's links, up to hi; j0: the item of w.
    template <uint32_t U>
    __device__ __forceinline__ void kill_window(uint32_t w, uint32_t hi, uint32_t &j0) {
        const uint32_t lane = threadIdx.x & 31, par = round & 1u;
        uint32_t ed[U], ts[U];
        uint2 l[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            const uint32_t x = w + 32u * u + lane, j = dev::items_of(s.off, s.n, w + 32u * u, j0);
            ed[u] = s.id[j];
            l[u] = x < hi ? *entry(j, x) : make_uint2(0u, 0u);
        }
        uint32_t kB[U], first[U];
        bool die[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            const bool act = w + 32u * u + lane < hi;
            ts[u] = !act ? 0u : l[u].x >> 31 ? 2u : twin_state(l[u].x - e0);
            // died earlier; or both edges in the batch: counted by the smaller id
            die[u] = ts[u] == 2u || (ts[u] == 1u && ed[u] < l[u].x - e0);
            first[u] = 1u;
            kB[u] = 0;
            if (die[u]) {
                // k_B and the count of deaths in one word: one access
                const unsigned long long old =
                    atomicAdd(reinterpret_cast<unsigned long long *>(&a.bl[l[u].y].k), 1ull << 32);
                kB[u] = (uint32_t)old;
                first[u] = (uint32_t)(old >> 32);
            }
        }
        uint32_t tw[U];
        int dec[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            tw[u] = l[u].x - e0;
            dec[u] = 0;
            if (!die[u]) continue;
            if (ts[u] == 2u && kB[u] > 1u) {
                upd += l[u].x != kAssigned;
                if (!(l[u].x >> 31)) dec[u] = (int)(kB[u] - 1u);
            }
        }
        // blooms touched for the first time: one counter atomic a warp
        uint32_t nf = 0;
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) nf += first[u] == 0u;
        const uint32_t incl = dev::warp_incl_scan(nf), sum = __shfl_sync(kAll, incl, 31);
        if (sum) {
            uint32_t q = 0, g = 0;
            if (lane == 0) {
                q = atomicAdd(&s.nt[par], sum);
                const uint32_t over = q + sum <= kTouch ? 0u : q >= kTouch ? sum : q + sum - kTouch;
                if (over) g = atomicAdd(&s0.nover[par], over);
            }
            q = __shfl_sync(kAll, q, 0);
            g = __shfl_sync(kAll, g, 0) - (q < kTouch ? kTouch : q);  // place of entry x >= kTouch: g + x
            q += incl - nf;
#pragma unroll
            for (uint32_t u = 0; u < U; ++u) {
                if (first[u]) continue;
                if (q < kTouch) s.touch[q] = l[u].y;
                else a.touch[b0 + g + q] = l[u].y;
                ++q;
            }
        }
        lose<U>(tw, dec);
    }

    // Phase 1: the links of the batch [head, head + F).
    __device__ __forceinline__ void kill_batch(uint32_t head, uint32_t F) {
        const uint32_t tid = threadIdx.x, par = round & 1u;
        if constexpr (kS) {
            mark(head, F, kBatch);
            if (F > kNT) __syncthreads();  // (lay's barrier does for one turn)
        }
        for (uint32_t c0 = 0; c0 < F;) {
            uint32_t n = F - c0 < kNT ? F - c0 : kNT;
            const uint32_t i = c0 + tid;
            uint32_t e = 0, d = 0;
            unsigned long long lb = 0;
            if (tid < n) {
                uint4 r;  // first link, links
                if (!kC && i < kFront) {
                    e = s.fe[par][i];
                    r = s.front[par][i];
                } else {
                    e = __ldcg(&a.fq[e0 + head + i]);
                    r = a.er[e0 + e];
                }
                lb = (unsigned long long)r.y << 32 | r.x;
                d = r.z;
            }
            unsigned long long total = lay(n, d, e, 0u, a.inc + lb);
            if (total >> 31) {  // too many links for one turn: one edge
                __syncthreads();
                n = 1;
                total = lay(n, tid == 0 ? d : 0u, e, 0u, a.inc + lb);
            }
            c0 += n;
            // a block peels on the blooms it touches: when there are fewer links
            // than threads, neighbouring shares go to different blocks (else the
            // first blocks had all the blooms of a small batch; the last part of a
            // 2M-edge graph, 1,516 rounds by a cluster, went from 77 to 53 ms)
            const uint32_t warp =
                total < (uint64_t)nranks * kNT ? (tid >> 5) * nranks + rank : rank * (kNT / 32) + (tid >> 5);
            uint32_t lo, hi;
            dev::share_of((uint32_t)total, warp, nranks * (kNT / 32), lo, hi);
            uint32_t j0 = lo < hi ? dev::item_of(s.off, s.n, lo) : 0u;
            if (hi - lo > 32u) {
                for (uint32_t w = lo; w < hi; w += 32u * kU) kill_window<kU>(w, hi, j0);
            } else if (lo < hi) {
                kill_window<1>(lo, hi, j0);
            }
            if (c0 < F) __syncthreads();  // the tables are laid anew
        }
    }

    // Entries [w, w + 32 U) of the touched blooms' pairs, up to hi.
    template <uint32_t U>
    __device__ __forceinline__ void apply_window(uint32_t w, uint32_t hi, uint32_t &j0) {
        const uint32_t lane = threadIdx.x & 31;
        uint2 pr[U];
        uint32_t c[U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            const uint32_t x = w + 32u * u + lane, j = dev::items_of(s.off, s.n, w + 32u * u, j0);
            c[u] = s.c[j];
            pr[u] = x < hi ? *entry(j, x) : make_uint2(0u, 0u);
        }
        uint32_t ed[2 * U];
        int dec[2 * U];
#pragma unroll
        for (uint32_t u = 0; u < U; ++u) {
            const bool act = w + 32u * u + lane < hi;
            const uint32_t x = pr[u].x - e0, y = pr[u].y - e0;
            const bool al = act && (pr[u].x >> 31 || remains(x)) && (pr[u].y >> 31 || remains(y));
            if (al) upd -= (pr[u].x == kAssigned) + (pr[u].y == kAssigned);
            ed[2 * u] = x;
            ed[2 * u + 1] = y;
            dec[2 * u] = al && !(pr[u].x >> 31) ? (int)c[u] : 0;
            dec[2 * u + 1] = al && !(pr[u].y >> 31) ? (int)c[u] : 0;
        }
        lose<2 * U>(ed, dec);
    }

    // Phase 2: n touched blooms, B for thread tid < n.
    __device__ __forceinline__ void apply_blooms(uint32_t n, uint32_t B) {
        const uint32_t tid = threadIdx.x;
        uint4 r = make_uint4(0u, 0u, 0u, 0u);  // first pair, pairs, k_B, C(B)
        if (tid < n) r = __ldcg(reinterpret_cast<const uint4 *>(a.bl + B));
        // nothing remains of a bloom whose pairs all died
        const uint32_t total =
            (uint32_t)lay(n, r.z != r.w ? r.y : 0u, B, r.w, r.y <= 2u ? a.bl[B].pair : a.pairs + r.x);
        uint32_t lo, hi;
        dev::share_of(total, tid >> 5, kNT / 32, lo, hi);
        uint32_t j0 = lo < hi ? dev::item_of(s.off, s.n, lo) : 0u;
        if (hi - lo > 32u) {
            for (uint32_t w = lo; w < hi; w += 32u * kU) apply_window<kU>(w, hi, j0);
        } else if (lo < hi) {
            apply_window<1>(lo, hi, j0);
        }
        __syncthreads();  // the tables are free again
        if (tid < n) {
            *reinterpret_cast<uint2 *>(&a.bl[B].k) = make_uint2(r.z - r.w, 0u);
            if (r.z != r.w) {
                upd += 2ull * (r.z - r.w);
                if (a.assigned) upd -= r.y <= 2u ? r.x : __ldcg(&a.bl[B].pair[0].x);
            }
            slots += r.y;
        }
    }

    // Level jump: k becomes the minimum support, the batch every edge at it.
    // By block 0 (of a cluster).
    __device__ void jump(uint32_t &na, uint32_t &ap) {
        const int tid = threadIdx.x, lane = tid & 31;
        uint32_t nn = s.nn[cur], ce = 0;
        int best = INT_MAX, cs = INT_MAX;  // this thread's entry of the first kNT
        for (uint32_t i = tid; i < nn; i += kNT) {
            const uint32_t e = __ldcg(&a.near[cur][e0 + i]);
            const int v = alive_sup(e);
            if (v >= 0) {
                best = v < best ? v : best;
                if (i < kNT) {
                    ce = e;
                    cs = v;
                }
            }
        }
        unsigned long long scan = tid == 0 ? nn : 0;
        best = warp_min(best);
        if (lane == 0 && best != INT_MAX) atomicMin(&s.mn, best);
        __syncthreads();
        int mn = s.mn;
        const bool rebuild = mn == INT_MAX;
        if (rebuild) {
            __syncthreads();  // everyone has read s.mn
            if (tid == 0) scan += 2ull * na;
            for (uint32_t i0 = 0; i0 < na; i0 += kNT) {
                const uint32_t i = i0 + tid;
                uint32_t e = 0;
                bool keep = false;
                if (i < na) {
                    e = __ldcg(&a.alive[ap][e0 + i]);
                    const int v = alive_sup(e);
                    keep = v >= 0;
                    if (keep) best = v < best ? v : best;
                }
                const uint32_t q = warp_place(&s.na, keep, lane);
                if (keep) a.alive[ap ^ 1u][e0 + q] = e;
            }
            best = warp_min(best);
            if (lane == 0 && best != INT_MAX) atomicMin(&s.mn, best);
            __syncthreads();
            mn = s.mn;
            na = s.na;
            ap ^= 1u;
            khi = window_top(mn);
        }
        k = mn > k ? mn : k;
        // the batch, and the window entries that stay
        const uint32_t cnt = rebuild ? na : nn;
        const uint32_t *src = rebuild ? a.alive[ap] : a.near[cur];
        for (uint32_t i0 = 0; i0 < cnt; i0 += kNT) {
            const uint32_t i = i0 + tid;
            uint32_t e = 0;
            int v = INT_MAX;
            if (!rebuild && i0 == 0) {
                e = ce;
                v = cs;
            } else if (i < cnt) {
                e = __ldcg(&src[e0 + i]);
                v = alive_sup(e);
                if (v < 0) v = INT_MAX;
            }
            const bool take = v <= k, keep = !take && v < khi;
            const uint32_t qs = warp_place(&s.sel, take, lane);
            if (take) settle(e, round, tail, qs);
            const uint32_t qn = warp_place(&s.nn[cur ^ 1u], keep, lane);
            if (keep) a.near[cur ^ 1u][e0 + qn] = e;
        }
        if constexpr (!kC) copies_done();
        __syncthreads();
        tail += s.sel;
        cur ^= 1u;
        if (scan) atomicAdd(&a.stats[2], scan);
    }

    __device__ void run(uint32_t ne) {
        const uint32_t tid = threadIdx.x, lane = tid & 31;
        for (uint32_t i = rank * kNT + tid; i < ne; i += nranks * kNT) {
            sup[i] = (int)a.er[e0 + i].w;
            if constexpr (!kS) st[i] = kAlive;
            a.alive[0][e0 + i] = i;
        }
        if (tid == 0) {
            s.nj[0] = s.nj[1] = s.nover[0] = s.nover[1] = s.nt[0] = s.nt[1] = 0;
            s.nn[0] = s.nn[1] = s.na = s.sel = 0;
            s.mn = INT_MAX;
        }
        barrier();
        uint32_t head = 0, na = ne, ap = 0, lvl = 0;
        for (;;) {
            if (head == tail) {
                if (rank == 0 && tid == 0 && lvl) atomicMax(&a.depth[k], lvl);
                if (tail == ne) break;
                lvl = 0;
                if (!kC || rank == 0) jump(na, ap);
                if constexpr (kC) {
                    if (rank == 0 && tid == 0) {
                        s.k = k;
                        s.khi = khi;
                        s.tail = tail;
                        s.cur = cur;
                    }
                    barrier();
                    k = s0.k;
                    khi = s0.khi;
                    tail = s0.tail;
                    cur = s0.cur;
                }
            }
            if (round > a.round_limit) {
                if (tid == 0) atomicOr(a.err, 2u);
                break;
            }
            const uint32_t par = round & 1u;
            kill_batch(head, tail - head);
            barrier();
            const uint32_t nt = s.nt[par] < kTouch ? s.nt[par] : kTouch, nover = s0.nover[par];
            if (tid == 0) {
                // what the next round and the next level jump start from
                s.nt[par ^ 1u] = 0;
                if (rank == 0) {
                    s.nj[par ^ 1u] = s.nover[par ^ 1u] = 0;
                    s.nn[cur ^ 1u] = s.na = s.sel = 0;
                    s.mn = INT_MAX;
                }
            }
            if constexpr (kS) mark(head, tail - head, kDead);
            for (uint32_t c0 = 0; c0 < nt; c0 += kNT)
                apply_blooms(nt - c0 < kNT ? nt - c0 : kNT, c0 + tid < nt ? s.touch[c0 + tid] : 0u);
            const uint32_t o1 = (uint32_t)((uint64_t)nover * (rank + 1u) / nranks);
            for (uint32_t c0 = (uint32_t)((uint64_t)nover * rank / nranks); c0 < o1; c0 += kNT) {
                const uint32_t B = c0 + tid < o1 ? __ldcg(&a.touch[b0 + c0 + tid]) : 0u;
                apply_blooms(o1 - c0 < kNT ? o1 - c0 : kNT, B);
            }
            barrier();
            head = tail;
            tail += s0.nj[par];
            ++round;
            ++lvl;
        }
        upd = dev::warp_sum(upd);
        slots = dev::warp_sum(slots);
        if (lane == 0) {
            if (upd) atomicAdd(&a.stats[0], upd);
            if (slots) atomicAdd(&a.stats[1], slots);
        }
    }
};

template <bool kC>
__global__ void __launch_bounds__(kNT, 1) k_peel_parts(const __grid_constant__ LocalArgs a) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    Shared &s = *reinterpret_cast<Shared *>(s_dyn);
    Shared *s0 = &s;
    uint32_t rank = 0, nranks = 1;
    if constexpr (kC) {
        cg::cluster_group c = cg::this_cluster();
        rank = c.block_rank();
        nranks = c.num_blocks();
        s0 = c.map_shared_rank(&s, 0);
    }
    for (;;) {
        if constexpr (kC) cg::this_cluster().sync();
        else __syncthreads();
        if (rank == 0 && threadIdx.x == 0) s.part = atomicAdd(a.queue, 1u);
        if constexpr (kC) cg::this_cluster().sync();
        else __syncthreads();
        const uint32_t i = s0->part;
        if (i >= a.np) break;
        const uint32_t p = a.order ? a.order[i] : a.np - 1u - i;
        const uint32_t e0 = a.part_e[p], ne = a.part_e[p + 1] - e0, b0 = a.part_b[p];
        if (ne == 0) continue;
        if constexpr (kC) {
            Part<true> P{a, s, *s0, e0, b0, rank, nranks, a.sup + e0, a.st + e0};
            P.run(ne);
        } else {  // ne <= kCap
            Part<false> P{a, s, s, e0, b0, 0u, 1u, reinterpret_cast<int *>(s_dyn + sizeof(Shared)), nullptr};
            P.run(ne);
        }
    }
    if constexpr (kC) cg::this_cluster().sync();  // no block leaves while another reads its shared memory
}

// Rounds (sum of the levels' depths), levels and the largest level.
__global__ void k_depth_sum(const uint32_t *depth, uint64_t m, unsigned long long *out) {
    unsigned long long r = 0, l = 0, top = 0;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i <= m; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t d = depth[i];
        r += d;
        l += d != 0;
        if (d) top = i;
    }
    r = dev::warp_sum(r);
    l = dev::warp_sum(l);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(kAll, top, o);
        top = y > top ? y : top;
    }
    if ((threadIdx.x & 31) == 0 && r) {
        atomicAdd(&out[0], r);
        atomicAdd(&out[1], l);
        atomicMax(&out[2], top);
    }
}

__global__ void k_unplace(const uint32_t *phi, const uint32_t *out_id, uint64_t first, uint64_t m, uint32_t *out) {
    for (uint64_t i = first + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x)
        out[out_id[i]] = phi[i];
}

inline unsigned grid_for(uint64_t items, int threads, unsigned cap) {
    uint64_t g = (items + threads - 1) / threads;
    if (g == 0) g = 1;
    return (unsigned)(g < cap ? g : cap);
}

}  // namespace

cudaError_t peel_parts(const PartGraph &g, uint32_t *phi_out, long long assign_from, PeelResult &res, int num_sms,
                       Alloc &al) {
    const uint64_t m = g.m;
    res = PeelResult{};
    if (m == 0) return cudaSuccess;
    struct Head {
        unsigned long long stats[3], sums[3];
        uint32_t queue, heavy_queue, err;
    };
    LocalArgs a{};
    a.part_e = g.part_e;
    a.part_b = g.part_b;
    a.order = g.order;
    a.np = g.np;
    a.er = g.er;
    a.inc = g.inc;
    a.pairs = g.pairs;
    a.bl = g.bl;
    if (g.n_heavy) {
        a.sup = al.get<int>(m);
        a.st = al.get<uint32_t>(m);
    }
    a.fq = al.get<uint32_t>(m);
    for (int i = 0; i < 2; ++i) {
        a.near[i] = al.get<uint32_t>(m);
        a.alive[i] = al.get<uint32_t>(m);
    }
    a.touch = al.get<uint32_t>(g.nb);
    a.phi = g.out_id ? al.get<uint32_t>(m) : phi_out;
    const uint64_t deep = g.deep;  // levels are below it
    a.depth = al.get<uint32_t>(deep + 1);
    Head *hd = al.get<Head>(1);
    if (al.err != cudaSuccess) return al.err;
    a.stats = hd->stats;
    a.err = &hd->err;
    a.assign_from = assign_from;
    a.assigned = g.assigned;
    a.queue = &hd->queue;
    const bt_limits *lim = al.limits;
    a.round_limit = lim && lim->peel_round_limit && lim->peel_round_limit < deep + 1 ? lim->peel_round_limit : deep + 1;
    cudaStream_t st = al.stream;
    BT_CUDA(cudaMemsetAsync(hd, 0, sizeof(Head), st));
    BT_CUDA(cudaMemsetAsync(a.depth, 0, sizeof(uint32_t) * (deep + 1), st));
    if (g.out_id && assign_from > 0) BT_CUDA(cudaMemsetAsync(a.phi, 0xFF, sizeof(uint32_t) * m, st));
    Forked side(*al.side, st);
    if (g.n_heavy) {
        // the heavy parts, each by a cluster of blocks, beside the kernel of the
        // others, which fills the rest of the SMs
        BT_CUDA(side.fork());
        const int smem = (int)sizeof(Shared);
        BT_CUDA(cudaFuncSetAttribute(k_peel_parts<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        BT_CUDA(cudaFuncSetAttribute(k_peel_parts<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = kCluster;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        cfg.blockDim = dim3(kNT);
        cfg.gridDim = dim3(kCluster);
        cfg.dynamicSmemBytes = sizeof(Shared);
        cfg.stream = al.side->stream;
        int nc = 0;
        BT_CUDA(cudaOccupancyMaxActiveClusters(&nc, k_peel_parts<true>, &cfg));
        if (nc > num_sms / (int)kCluster) nc = num_sms / (int)kCluster;
        if (nc < 1) nc = 1;
        if ((uint32_t)nc > g.n_heavy) nc = (int)g.n_heavy;
        cfg.gridDim = dim3(kCluster * (unsigned)nc);
        LocalArgs h = a;
        h.np = g.n_heavy;
        h.queue = &hd->heavy_queue;
        BT_CUDA(cudaLaunchKernelEx(&cfg, k_peel_parts<true>, h));
        al.launches++;
        a.order = g.order + g.n_heavy;
        a.np = g.np - g.n_heavy;
    }
    if (a.np) {
        const size_t smem = sizeof(Shared) + sizeof(int) * kCap;
        BT_CUDA(cudaFuncSetAttribute(k_peel_parts<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        const unsigned grid = (unsigned)num_sms < a.np ? (unsigned)num_sms : a.np;
        k_peel_parts<false><<<grid, kNT, smem, st>>>(a);
        al.launches++;
    }
    BT_CUDA(side.join());
    if (g.out_id) {
        k_unplace<<<grid_for(m - g.first_e, 256, (unsigned)num_sms * 16), 256, 0, st>>>(a.phi, g.out_id, g.first_e, m, phi_out);
        al.launches++;
    }
    k_depth_sum<<<grid_for(deep + 1, 256, (unsigned)num_sms * 8), 256, 0, st>>>(a.depth, deep, hd->sums);
    al.launches++;
    BT_CUDA(cudaGetLastError());
    Head h{};
    BT_CUDA(cudaMemcpyAsync(&h, hd, sizeof(Head), cudaMemcpyDeviceToHost, st));
    BT_CUDA(cudaStreamSynchronize(st));
    res.rounds = h.sums[0];
    res.levels = h.sums[1];
    res.kmax = h.sums[2];
    res.updates = h.stats[0];
    res.slots = h.stats[1];
    res.scanned = h.stats[2];
    // the same line as the grid kernel's: rounds 0 .. round_limit may run
    if (h.err || res.rounds > a.round_limit + 1) res.status = BT_ERR_NOCONVERGE;
    al.put(a.sup);
    al.put(a.st);
    al.put(a.fq);
    for (int i = 0; i < 2; ++i) {
        al.put(a.near[i]);
        al.put(a.alive[i]);
    }
    al.put(a.touch);
    if (g.out_id) al.put(a.phi);
    al.put(a.depth);
    al.put(hd);
    return cudaSuccess;
}

}  // namespace bt
