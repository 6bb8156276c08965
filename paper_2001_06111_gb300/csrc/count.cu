// Butterfly support counting and BE-Index construction by priority-obeyed
// wedge enumeration (Section IV-B, Alg. 3; Defs. 7, 8, 10).
//
// For a start vertex u (processed in rank space, so p(x) < p(u) <=> x < u):
//   pass A  for v in N(u), v < u; for w in N(v), w < u:  cnt[w] += 1
//           -> cnt[w] = |N(u) ∩ N(w) ∩ {x < u}|  (Alg. 3, the first wedge loop)
//   pass B  every wedge (u,v,w) with c = cnt[w] >= 2 lies in the maximal
//           priority-obeyed bloom anchored by (u,w), a c-bloom (Lemma 7); each
//           of its two edges is in c-1 of the bloom's butterflies (Lemma 2)
//           and every butterfly lies in exactly one such bloom (Lemma 3), so
//           support(u,v) += c-1 and support(v,w) += c-1 sums to the support.
//   emit    the bloom gets bloom number c, and the wedge becomes one twin
//           pair ((u,v),(v,w)) linked to it (Alg. 3, the second wedge loop).
//
// Counting (k_count, k_count_light).  Start vertices with few wedges are counted
// by a warp with a hash table in shared memory; the others by a block, heaviest
// first.  A block lays the wedges over up to 1,024 middle vertices side by side
// (dev::items_of), so every lane has four wedges in flight whatever the degrees.
// What bounded the dense counters of a block in global memory was the rate of
// scattered accesses (3 GB of them on the 30M-edge graph): now the counters of the
// vertices ranked just below the start vertex, the ones most wedges end at, are in
// shared memory, and only those of lower ones are in global memory.  Wedges end in
// the layer they start from, so on graphs with more vertices than counters there
// the counters go by places in the layer: by rank, half of them were of the other
// layer.  Wedges that end below the window: 48 to 35 % at 30M edges, 23 to 7 % at
// 2M; counting 30M edges 320 -> 151 -> 132 ms, building the index of 2M edges 20.4
// -> 11.2 -> 9.6.  What bounds it at 30M edges are those accesses; at 3M the shared
// memory path is busy 57 % of the time and the issue slots 41 %.
#include "bt_device.cuh"
#include "bt_internal.cuh"

namespace bt {
namespace {

__device__ __forceinline__ uint32_t ld_cg(const uint32_t *p) { return __ldcg(p); }

// ------------------------------------------------------------------- count
constexpr int kCT = 1024;                // threads of a count block (one an SM)
constexpr uint32_t kCU = 4;              // wedges a lane has in flight
constexpr uint32_t kHot = 88 * 1024;     // 16-bit counters in shared memory

struct CountArgs {
    const uint64_t *off;
    const uint32_t *adj, *eid, *hv, *pl;
    const uint32_t *wend, *place;  // what counters go by: places in a layer, or adj and null
    const uint64_t *wv;
    uint32_t lo, hi;
    const uint32_t *heavy, *n_heavy;
    const uint32_t *vbase;
    uint32_t cold_n;  // 32-bit counters of a block in global memory
    uint32_t *cold;
    unsigned long long *support;
    uint32_t *inc_cnt;
    uint64_t *w2v, *nbv;
    unsigned long long *totals;  // sum of c - 1 over bloom wedges: twice the butterflies
    uint32_t *queue;
    const uint8_t *assigned;
};

struct CountShared {
    uint32_t n;
    uint32_t off[kCT + 1];           // first wedge of each middle vertex
    uint32_t e[kCT + 1];             // its edge (u, v)
    unsigned long long at[kCT + 1];  // wedge x of item j is arc at[j] + x
    uint32_t acc[kCT + 1], inc[kCT + 1];  // support and links of (u, v) from these (supports are below m < 2^31)
    uint32_t u;
};
// lanes past the last wedge get item n (dev::items_of), which has a place in every table
static_assert(sizeof(CountShared::e) == sizeof(CountShared::off) && sizeof(CountShared::acc) == sizeof(CountShared::off) &&
                  sizeof(CountShared::inc) == sizeof(CountShared::off) &&
                  sizeof(CountShared::at) == 2 * sizeof(CountShared::off),
              "tables of kCT items and one more");

// Lays the wedges over middle vertices [c0, c0 + kCT) of u side by side, empty
// ones left out.  Returns their number.
__device__ __forceinline__ uint32_t lay_wedges(CountShared &s, const CountArgs &a, uint64_t arc, uint32_t h, uint32_t c0) {
    const uint32_t tid = threadIdx.x, i = c0 + tid;
    uint32_t len = 0, e = 0;
    uint64_t at = 0;
    if (i < h) {
        len = a.pl[arc + i];
        if (len) {
            e = a.eid[arc + i];
            at = a.off[a.adj[arc + i]];
        }
    }
    unsigned long long all;
    const unsigned long long ex =
        dev::block_excl_scan<unsigned long long>((unsigned long long)(len > 0u) << 48 | len, &all);
    const uint32_t j = (uint32_t)(ex >> 48), x = (uint32_t)ex;
    if (len) {
        s.off[j] = x;
        s.e[j] = e;
        s.at[j] = at - x;
    }
    if (tid == kCT - 1) {
        s.n = j + (len > 0u);
        s.off[j + (len > 0u)] = (uint32_t)all;
    }
    __syncthreads();
    return (uint32_t)all;
}

// Start vertices with many wedges, one block each, heaviest first.  The counters
// of the kHot places below u are in shared memory (they ascend with degree, so
// they are met by most wedges of a skewed graph), 16 bits each; a start vertex of
// 2^16 or more middle vertices uses half the ranks with 32 bits.  Those of lower
// ranks are 32-bit words of this block in global memory: when a count fits 16
// bits its readers in pass B are counted in the high half and the last one
// clears the word, else a third walk clears them.
template <bool kIndex>
__global__ void __launch_bounds__(kCT) k_count(const __grid_constant__ CountArgs a) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    CountShared &s = *reinterpret_cast<CountShared *>(s_dyn);
    uint32_t *hot = reinterpret_cast<uint32_t *>(s_dyn + sizeof(CountShared));
    uint32_t *cold = a.cold + (size_t)blockIdx.x * a.cold_n;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (uint32_t i = tid; i < kHot / 2; i += kCT) hot[i] = 0;
    s.acc[tid] = 0;
    s.inc[tid] = 0;
    unsigned long long twice = 0;
    const uint32_t n_heavy = a.n_heavy[64];
    if (tid == 0) s.u = atomicAdd(a.queue, 1u);
    __syncthreads();
    for (;;) {
        const uint32_t q = s.u;
        if (q >= n_heavy) break;
        __syncthreads();
        uint32_t next = 0;  // the following turn, asked for ahead
        if (tid == 0) next = atomicAdd(a.queue, 1u);
        const uint32_t u = a.heavy[q];
        if (u >= a.lo && u < a.hi) {
            const uint64_t arc = a.off[u];
            const uint32_t h = a.hv[u];
            const uint32_t vb = a.vbase ? a.vbase[u] : 0u;
            const bool narrow = h < 0x10000u;  // a count never exceeds h
            const uint32_t width = narrow ? kHot : kHot / 2;
            const uint32_t ru = a.place ? a.place[u] : u - vb;
            const uint32_t base = ru > width ? ru - width : 0u;  // hot counters are those of ranks [base, ru)
            unsigned long long w2 = 0, nb = 0;
            // pass A: cnt[w] += 1; the second wedge of an end vertex makes its bloom
            for (uint32_t c0 = 0; c0 < h; c0 += kCT) {
                const uint32_t total = lay_wedges(s, a, arc, h, c0);
                uint32_t lo, hi;
                dev::share_of(total, warp, kCT / 32, lo, hi);
                uint32_t j0 = lo < hi ? dev::item_of(s.off, s.n, lo) : 0u;
                for (uint32_t x0 = lo; x0 < hi; x0 += 32u * kCU) {
                    uint32_t w[kCU], old[kCU];
#pragma unroll
                    for (uint32_t r = 0; r < kCU; ++r) {
                        const uint32_t x = x0 + 32u * r + lane, j = dev::items_of(s.off, s.n, x0 + 32u * r, j0);
                        w[r] = x < hi ? a.wend[s.at[j] + x] - vb : 0xFFFFFFFFu;
                    }
#pragma unroll
                    for (uint32_t r = 0; r < kCU; ++r) {
                        old[r] = 0;
                        if (w[r] == 0xFFFFFFFFu) continue;
                        if (w[r] >= base) {
                            const uint32_t i = w[r] - base;
                            if (narrow) old[r] = atomicAdd(&hot[i >> 1], 1u << (16u * (i & 1u))) >> (16u * (i & 1u)) & 0xFFFFu;
                            else old[r] = atomicAdd(&hot[i], 1u);
                        } else if (kIndex) {
                            old[r] = atomicAdd(&cold[w[r]], 1u);
                        } else {
                            atomicAdd(&cold[w[r]], 1u);
                        }
                    }
                    if (kIndex) {
#pragma unroll
                        for (uint32_t r = 0; r < kCU; ++r) nb += old[r] == 1u;
                    }
                }
                __syncthreads();
            }
            // pass B: attribute c - 1 to both edges of every wedge in a bloom
            for (uint32_t c0 = 0; c0 < h; c0 += kCT) {
                const uint32_t total = lay_wedges(s, a, arc, h, c0);
                uint32_t lo, hi;
                dev::share_of(total, warp, kCT / 32, lo, hi);
                uint32_t j0 = lo < hi ? dev::item_of(s.off, s.n, lo) : 0u;
                for (uint32_t x0 = lo; x0 < hi; x0 += 32u * kCU) {
                    uint32_t w[kCU], c[kCU], jj[kCU], e[kCU];
#pragma unroll
                    for (uint32_t r = 0; r < kCU; ++r) {
                        const uint32_t x = x0 + 32u * r + lane;
                        jj[r] = dev::items_of(s.off, s.n, x0 + 32u * r, j0);
                        w[r] = x < hi ? a.wend[s.at[jj[r]] + x] - vb : 0xFFFFFFFFu;
                    }
#pragma unroll
                    for (uint32_t r = 0; r < kCU; ++r) {
                        c[r] = 0;
                        if (w[r] == 0xFFFFFFFFu) continue;
                        if (w[r] >= base) {
                            const uint32_t i = w[r] - base;
                            c[r] = narrow ? hot[i >> 1] >> (16u * (i & 1u)) & 0xFFFFu : hot[i];
                        } else if (narrow) {
                            const uint32_t old = atomicAdd(&cold[w[r]], 1u << 16);
                            c[r] = old & 0xFFFFu;
                            if ((old >> 16) + 1u == c[r]) cold[w[r]] = 0u;  // every wedge has read it
                        } else {
                            c[r] = ld_cg(&cold[w[r]]);
                        }
                    }
#pragma unroll
                    for (uint32_t r = 0; r < kCU; ++r) {
                        const uint32_t x = x0 + 32u * r + lane;
                        e[r] = c[r] >= 2u ? a.eid[s.at[jj[r]] + x] : 0u;
                    }
#pragma unroll
                    for (uint32_t r = 0; r < kCU; ++r) {
                        if (c[r] < 2u) continue;
                        atomicAdd(&a.support[e[r]], (unsigned long long)(c[r] - 1u));
                        atomicAdd(&s.acc[jj[r]], c[r] - 1u);
                        twice += c[r] - 1u;
                        if (kIndex) {
                            // edges already assigned (progressive compression) get no links
                            if (!a.assigned || !a.assigned[e[r]]) atomicAdd(&a.inc_cnt[e[r]], 1u);
                            atomicAdd(&s.inc[jj[r]], 1u);
                            ++w2;
                        }
                    }
                }
                __syncthreads();
                if (tid < s.n) {
                    const uint32_t e = s.e[tid];
                    if (s.acc[tid]) atomicAdd(&a.support[e], (unsigned long long)s.acc[tid]);
                    s.acc[tid] = 0;
                    if (kIndex && s.inc[tid]) {
                        if (!a.assigned || !a.assigned[e]) atomicAdd(&a.inc_cnt[e], s.inc[tid]);
                        s.inc[tid] = 0;
                    }
                }
                __syncthreads();
            }
            if (!narrow && base) {
                for (uint32_t c0 = 0; c0 < h; c0 += kCT) {
                    const uint32_t total = lay_wedges(s, a, arc, h, c0);
                    uint32_t lo, hi;
                    dev::share_of(total, warp, kCT / 32, lo, hi);
                    uint32_t j0 = lo < hi ? dev::item_of(s.off, s.n, lo) : 0u;
                    for (uint32_t x0 = lo; x0 < hi; x0 += 32u) {
                        const uint32_t x = x0 + lane, j = dev::items_of(s.off, s.n, x0, j0);
                        const uint32_t w = x < hi ? a.wend[s.at[j] + x] - vb : 0xFFFFFFFFu;
                        if (w < base) cold[w] = 0u;
                    }
                    __syncthreads();
                }
            }
            const uint32_t used = narrow ? (ru - base + 1u) / 2u : ru - base;
            for (uint32_t i = tid; i < used; i += kCT) hot[i] = 0;
            if (kIndex) {
                const unsigned long long w2s = dev::block_sum(w2);
                const unsigned long long nbs = dev::block_sum(nb);
                if (tid == 0) {
                    a.w2v[u] = w2s;
                    a.nbv[u] = nbs;
                }
            }
        }
        if (tid == 0) s.u = next;
        __syncthreads();
    }
    twice = dev::block_sum(twice);
    if (tid == 0 && twice) atomicAdd(&a.totals[0], twice);
}

// Start vertices with few wedges, a warp each: the end vertices go to a hash
// table of the warp in shared memory.  Most start vertices of a skewed graph are
// of this kind; a block's barriers and its turn at the queue cost more than
// their wedges.
template <bool kIndex>
__global__ void __launch_bounds__(256) k_count_light(const __grid_constant__ CountArgs a) {
    constexpr uint32_t kSlots = 2 * kLightW, kWin = kLightW / 32, kWarps = 8;
    constexpr uint32_t kEmpty = 0xFFFFFFFFu;
    __shared__ uint32_t s_key[kWarps][kSlots], s_cnt[kWarps][kSlots];
    __shared__ uint32_t s_off[kWarps][33], s_acc[kWarps][32], s_inc[kWarps][32];
    __shared__ unsigned long long s_at[kWarps][33];
    const uint32_t lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    uint32_t *key = s_key[wi], *cnt = s_cnt[wi], *off = s_off[wi];
    for (uint32_t i = lane; i < kSlots; i += 32) {
        key[i] = kEmpty;
        cnt[i] = 0;
    }
    s_acc[wi][lane] = s_inc[wi][lane] = 0;
    __syncwarp();
    unsigned long long twice = 0;
    const uint32_t nw = gridDim.x * kWarps;
    // warp x takes ranks x, x + nw, ...: 32 looked up at a turn, so that a small
    // graph still gives every vertex its own warp
    const uint32_t ranks = a.hi - a.lo;
    for (uint64_t g = blockIdx.x * kWarps + wi; g < ranks; g += 32ull * nw) {
        bool light = false;
        uint32_t my_h = 0, my_u = 0;
        uint64_t my_arc = 0;
        if (g + (uint64_t)lane * nw < ranks) {
            const uint32_t u = my_u = a.lo + (uint32_t)(g + (uint64_t)lane * nw);
            const uint64_t W = a.wv[u];
            if (kIndex && W == 0) a.w2v[u] = a.nbv[u] = 0;
            if (W > 0) {
                my_h = a.hv[u];
                my_arc = a.off[u];
                light = is_light(W, my_h);
            }
        }
        unsigned todo = __ballot_sync(0xffffffffu, light);
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1u;
            const uint32_t u = __shfl_sync(0xffffffffu, my_u, src), h = __shfl_sync(0xffffffffu, my_h, src);
            const uint64_t arc = __shfl_sync(0xffffffffu, my_arc, src);
            uint32_t len = 0, e = 0;
            uint64_t at = 0;
            if (lane < h) {
                len = a.pl[arc + lane];
                if (len) {
                    e = a.eid[arc + lane];
                    at = a.off[a.adj[arc + lane]];
                }
            }
            const unsigned has = __ballot_sync(0xffffffffu, len > 0u);
            const uint32_t incl = dev::warp_incl_scan(len), total = __shfl_sync(0xffffffffu, incl, 31);
            const uint32_t j = __popc(has & ((1u << lane) - 1u)), n = __popc(has);
            if (len) {
                off[j] = incl - len;
                s_at[wi][j] = at - (incl - len);
            }
            if (lane == 31) off[n] = total;
            __syncwarp();
            uint32_t slot[kWin], jj[kWin], j0 = 0, nb = 0;
#pragma unroll
            for (uint32_t r = 0; r < kWin; ++r) {
                slot[r] = kEmpty;
                jj[r] = 0;
                if (32u * r < total) {
                    jj[r] = dev::items_of(off, n, 32u * r, j0);
                    const uint32_t x = 32u * r + lane;
                    if (x < total) slot[r] = a.adj[s_at[wi][jj[r]] + x];
                }
            }
#pragma unroll
            for (uint32_t r = 0; r < kWin; ++r) {
                if (slot[r] == kEmpty) continue;
                const uint32_t w = slot[r];
                uint32_t i = (w * 0x9E3779B1u) >> 23;  // 2^9 slots
                for (;;) {
                    const uint32_t k = atomicCAS(&key[i], kEmpty, w);
                    if (k == kEmpty || k == w) break;
                    i = (i + 1u) & (kSlots - 1u);
                }
                slot[r] = i;
                if (atomicAdd(&cnt[i], 1u) == 1u) ++nb;
            }
            __syncwarp();
            uint32_t w2 = 0;
#pragma unroll
            for (uint32_t r = 0; r < kWin; ++r) {
                if (slot[r] == kEmpty) continue;
                const uint32_t c = cnt[slot[r]];
                if (c < 2u) continue;
                const uint32_t ev = a.eid[s_at[wi][jj[r]] + 32u * r + lane];
                atomicAdd(&a.support[ev], (unsigned long long)(c - 1u));
                atomicAdd(&s_acc[wi][jj[r]], c - 1u);
                twice += c - 1u;
                if (kIndex) {
                    if (!a.assigned || !a.assigned[ev]) atomicAdd(&a.inc_cnt[ev], 1u);
                    atomicAdd(&s_inc[wi][jj[r]], 1u);
                    ++w2;
                }
            }
            __syncwarp();
            // the lane that read item j's record adds what the item gathered
            if (len) {
                const uint32_t acc = s_acc[wi][j];
                if (acc) atomicAdd(&a.support[e], (unsigned long long)acc);
                s_acc[wi][j] = 0;
                if (kIndex && s_inc[wi][j]) {
                    if (!a.assigned || !a.assigned[e]) atomicAdd(&a.inc_cnt[e], s_inc[wi][j]);
                    s_inc[wi][j] = 0;
                }
            }
#pragma unroll
            for (uint32_t r = 0; r < kWin; ++r)
                if (slot[r] != kEmpty) {
                    key[slot[r]] = kEmpty;
                    cnt[slot[r]] = 0;
                }
            if (kIndex) {
                w2 = dev::warp_sum(w2);
                nb = dev::warp_sum(nb);
                if (lane == 0) {
                    a.w2v[u] = w2;
                    a.nbv[u] = nb;
                }
            }
            __syncwarp();
        }
    }
    twice = dev::warp_sum(twice);
    if (lane == 0 && twice) atomicAdd(&a.totals[0], twice);
}

// -------------------------------------------------------------------- emit
// Emit the index: blooms (bloom number, first pair), twin pairs and the per-edge
// link lists, by the tiers and with the counters of the count kernels.  Once the
// counts of a start vertex are final, every end vertex w with two wedges or more
// gets a bloom: its id and the end of its pair range go to one 64-bit word, from
// whose low half each wedge takes its pair by an atomic.
//
// An edge is the first member of pairs of one start vertex only, its own higher
// endpoint: those links fill its list from the front, counted in shared memory.
// Links as second member come from many start vertices and fill it from the
// back, by one atomic on a 64-bit cursor an edge that starts at the list's end.
// What is left to bound it are the scattered 8-byte link stores and those cursors.
struct EmitArgs {
    CountArgs c;            // counters and graph (support, w2v, nbv unused)
    unsigned long long *word;  // [blocks * cnt_n] (pair range end | bloom << 32) of an end vertex
    uint32_t *found;        // [blocks * cold_n] end vertices below the hot ranks with a bloom
    uint32_t cnt_n;
    const uint64_t *bloom_base, *pair_base, *inc_off;
    unsigned long long *cursor;  // [m] end of the free places of each edge's list
    uint32_t *bloom_k, *bloom_off;
    uint2 *pairs, *inc;
    bool twin;
};

// A pair of bloom B in `slot`: euv is the first member, its link number `place`.
__device__ __forceinline__ void put_pair(const EmitArgs &a, uint32_t slot, uint32_t B, uint32_t euv, uint32_t evw,
                                         bool fu, bool fw, uint64_t at, unsigned long long back) {
    // an assigned edge is flagged in bit 31 and gets no link
    a.pairs[slot] = make_uint2(euv | (fu ? 0x80000000u : 0u), evw | (fw ? 0x80000000u : 0u));
    // each link carries its bloom and which member of the pair the edge is, or
    // the twin itself and the bloom
    if (!fu) a.inc[at] = make_uint2(a.twin ? evw : slot, B);
    if (!fw) a.inc[back - 1u] = make_uint2(a.twin ? euv : slot, B | (a.twin ? 0u : 0x80000000u));
}

struct EmitShared {
    CountShared c;
    unsigned long long front[kCT + 1];  // first free place of (u, v)'s list
    unsigned long long alloc;       // blooms (high) and pairs (low) of the start vertex handed out
    uint32_t n_found;
};
// From this many pairs a bloom on (the mean of a start vertex), windows of wedges go to
// the warps in turn, so that a bloom's pairs come to lie in the order of their middle
// vertices, whose edges are neighbours; by shares, 32 warps fill a bloom at once from
// 32 places of that order.  The peel of dense blooms reads and decrements along it
// (K_{1000,1000} 47 against 39 ms, a block of 1000 x 1000 of density 0.9 135
// against 107, of 300 x 300 2.7 against 2.2); where blooms have few pairs the
// order is worth nothing and finding the item of every window costs 7 % of emit (2M
// skewed edges 6.9 against 7.4 ms).
constexpr uint32_t kInTurn = 16;
// hot ranks of emit (its tables take more of the shared memory)
constexpr uint32_t kHotE = 80 * 1024;

// Blooms for the lanes whose end vertex w has c >= 2 wedges: id and pair range,
// one shared atomic a warp.
__device__ __forceinline__ void claim(const EmitArgs &a, unsigned long long *alloc, unsigned long long *word, uint32_t w,
                                      uint32_t c, uint64_t bb, uint64_t pb) {
    const uint32_t lane = threadIdx.x & 31;
    const bool has = c >= 2u;
    const unsigned m = __ballot_sync(0xffffffffu, has);
    if (!m) return;
    const uint32_t incl = dev::warp_incl_scan(has ? c : 0u), sum = __shfl_sync(0xffffffffu, incl, 31);
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(alloc, (unsigned long long)__popc(m) << 32 | sum);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (has) {
        const uint32_t B = (uint32_t)bb + (uint32_t)(base >> 32) + __popc(m & ((1u << lane) - 1u));
        const uint32_t end = (uint32_t)pb + (uint32_t)base + incl;
        a.bloom_k[B] = c;
        a.bloom_off[B] = end - c;
        word[w] = (unsigned long long)B << 32 | end;
    }
}

__global__ void __launch_bounds__(kCT) k_emit(const __grid_constant__ EmitArgs ea) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    EmitShared &es = *reinterpret_cast<EmitShared *>(s_dyn);
    CountShared &s = es.c;
    const CountArgs &a = ea.c;
    uint32_t *hot = reinterpret_cast<uint32_t *>(s_dyn + sizeof(EmitShared));
    uint32_t *cold = a.cold + (size_t)blockIdx.x * a.cold_n;
    uint32_t *found = ea.found + (size_t)blockIdx.x * a.cold_n;
    unsigned long long *word = ea.word + (size_t)blockIdx.x * ea.cnt_n;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (uint32_t i = tid; i < kHotE / 2; i += kCT) hot[i] = 0;
    const uint32_t n_heavy = a.n_heavy[64];
    if (tid == 0) s.u = atomicAdd(a.queue, 1u);
    __syncthreads();
    for (;;) {
        const uint32_t q = s.u;
        if (q >= n_heavy) break;
        __syncthreads();
        uint32_t next = 0;
        if (tid == 0) {
            next = atomicAdd(a.queue, 1u);
            es.alloc = 0;
            es.n_found = 0;
        }
        const uint32_t u = a.heavy[q];
        const uint64_t arc = a.off[u], bb = ea.bloom_base[u], pb = ea.pair_base[u];
        const uint32_t h = a.hv[u];
        const uint32_t vb = a.vbase ? a.vbase[u] : 0u;
        const bool narrow = h < 0x10000u;
        const uint32_t width = narrow ? kHotE : kHotE / 2;
        const uint32_t ru = a.place ? a.place[u] : u - vb;
        const uint32_t base = ru > width ? ru - width : 0u;
        __syncthreads();
        // counts, as in k_count; end vertices of lower ranks with a bloom are listed
        for (uint32_t c0 = 0; c0 < h; c0 += kCT) {
            const uint32_t total = lay_wedges(s, a, arc, h, c0);
            uint32_t lo, hi;
            dev::share_of(total, warp, kCT / 32, lo, hi);
            uint32_t j0 = lo < hi ? dev::item_of(s.off, s.n, lo) : 0u;
            for (uint32_t x0 = lo; x0 < hi; x0 += 32u * kCU) {
                uint32_t w[kCU], old[kCU];
#pragma unroll
                for (uint32_t r = 0; r < kCU; ++r) {
                    const uint32_t x = x0 + 32u * r + lane, j = dev::items_of(s.off, s.n, x0 + 32u * r, j0);
                    w[r] = x < hi ? a.wend[s.at[j] + x] - vb : 0xFFFFFFFFu;
                }
#pragma unroll
                for (uint32_t r = 0; r < kCU; ++r) {
                    old[r] = 0;
                    if (w[r] == 0xFFFFFFFFu) continue;
                    if (w[r] >= base) {
                        const uint32_t i = w[r] - base;
                        if (narrow) atomicAdd(&hot[i >> 1], 1u << (16u * (i & 1u)));
                        else atomicAdd(&hot[i], 1u);
                    } else {
                        old[r] = atomicAdd(&cold[w[r]], 1u);
                    }
                }
#pragma unroll
                for (uint32_t r = 0; r < kCU; ++r)
                    if (old[r] == 1u) found[atomicAdd(&es.n_found, 1u)] = w[r];
            }
            __syncthreads();
        }
        // blooms
        const uint32_t span = ru - base, n_found = es.n_found;
        for (uint32_t i0 = 0; i0 < span; i0 += kCT) {
            const uint32_t i = i0 + tid;
            const uint32_t c = i >= span ? 0u : narrow ? hot[i >> 1] >> (16u * (i & 1u)) & 0xFFFFu : hot[i];
            claim(ea, &es.alloc, word, base + i, c, bb, pb);
        }
        for (uint32_t i0 = 0; i0 < n_found; i0 += kCT) {
            const uint32_t i = i0 + tid, w = i < n_found ? found[i] : 0u;
            claim(ea, &es.alloc, word, w, i < n_found ? ld_cg(&cold[w]) : 0u, bb, pb);
        }
        __syncthreads();
        // every bloom wedge becomes a twin pair linked to both edges
        const bool in_turn = (uint32_t)es.alloc >= kInTurn * (uint32_t)(es.alloc >> 32);
        for (uint32_t c0 = 0; c0 < h; c0 += kCT) {
            const uint32_t total = lay_wedges(s, a, arc, h, c0);
            if (tid < s.n) {
                es.front[tid] = ea.inc_off[s.e[tid]];
                s.inc[tid] = a.assigned && a.assigned[s.e[tid]];
            }
            __syncthreads();
            uint32_t lo = warp * 32u * kCU, hi = total, j0 = 0;
            if (!in_turn) {
                dev::share_of(total, warp, kCT / 32, lo, hi);
                if (lo < hi) j0 = dev::item_of(s.off, s.n, lo);
            }
            for (uint32_t x0 = lo; x0 < hi; x0 += in_turn ? kCT * kCU : 32u * kCU) {
                if (in_turn) j0 = dev::item_of(s.off, s.n, x0);
                uint32_t w[kCU], jj[kCU], ev[kCU];
                unsigned long long wd[kCU], back[kCU], at[kCU];
                bool in[kCU];
#pragma unroll
                for (uint32_t r = 0; r < kCU; ++r) {
                    const uint32_t x = x0 + 32u * r + lane;
                    jj[r] = dev::items_of(s.off, s.n, x0 + 32u * r, j0);
                    w[r] = x < hi ? a.wend[s.at[jj[r]] + x] - vb : 0xFFFFFFFFu;
                }
#pragma unroll
                for (uint32_t r = 0; r < kCU; ++r) {
                    uint32_t c = 0;
                    if (w[r] != 0xFFFFFFFFu) {
                        if (w[r] >= base) {
                            const uint32_t i = w[r] - base;
                            c = narrow ? hot[i >> 1] >> (16u * (i & 1u)) & 0xFFFFu : hot[i];
                        } else {
                            c = ld_cg(&cold[w[r]]);
                            if (c == 1u) cold[w[r]] = 0u;  // its only reader
                        }
                    }
                    in[r] = c >= 2u;
                }
#pragma unroll
                for (uint32_t r = 0; r < kCU; ++r) {
                    wd[r] = in[r] ? atomicAdd(&word[w[r]], ~0ull) : 0ull;  // the low half is never 0: no borrow
                    ev[r] = in[r] ? a.eid[s.at[jj[r]] + x0 + 32u * r + lane] : 0u;
                }
                bool fu[kCU], fw[kCU];
#pragma unroll
                for (uint32_t r = 0; r < kCU; ++r) {
                    fu[r] = in[r] && s.inc[jj[r]] != 0u;
                    fw[r] = in[r] && a.assigned && a.assigned[ev[r]];
                    back[r] = in[r] && !fw[r] ? atomicAdd(&ea.cursor[ev[r]], ~0ull) : 0ull;
                    at[r] = in[r] && !fu[r] ? atomicAdd(&es.front[jj[r]], 1ull) : 0ull;
                }
#pragma unroll
                for (uint32_t r = 0; r < kCU; ++r)
                    if (in[r])
                        put_pair(ea, (uint32_t)wd[r] - 1u, (uint32_t)(wd[r] >> 32), s.e[jj[r]], ev[r], fu[r], fw[r],
                                 at[r], back[r]);
            }
            __syncthreads();
            if (tid < s.n) s.inc[tid] = 0;
            __syncthreads();
        }
        // counters back to zero
        for (uint32_t i = tid; i < n_found; i += kCT) cold[found[i]] = 0u;
        const uint32_t used = narrow ? (span + 1u) / 2u : span;
        for (uint32_t i = tid; i < used; i += kCT) hot[i] = 0;
        if (tid == 0) s.u = next;
        __syncthreads();
    }
}

// Start vertices with few wedges, a warp each (as k_count_light).
__global__ void __launch_bounds__(256) k_emit_light(const __grid_constant__ EmitArgs ea) {
    constexpr uint32_t kSlots = 2 * kLightW, kWin = kLightW / 32, kWarps = 8;
    constexpr uint32_t kEmpty = 0xFFFFFFFFu;
    __shared__ uint32_t s_key[kWarps][kSlots], s_cnt[kWarps][kSlots], s_bloom[kWarps][kSlots];
    __shared__ uint32_t s_off[kWarps][33], s_e[kWarps][32];
    __shared__ unsigned long long s_at[kWarps][33], s_front[kWarps][32];
    const CountArgs &a = ea.c;
    const uint32_t lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
    uint32_t *key = s_key[wi], *cnt = s_cnt[wi], *bloom = s_bloom[wi], *off = s_off[wi];
    for (uint32_t i = lane; i < kSlots; i += 32) {
        key[i] = kEmpty;
        cnt[i] = 0;
    }
    __syncwarp();
    const uint32_t nw = gridDim.x * kWarps, ranks = a.hi - a.lo;
    for (uint64_t g = blockIdx.x * kWarps + wi; g < ranks; g += 32ull * nw) {
        bool light = false;
        uint32_t my_h = 0, my_u = 0;
        if (g + (uint64_t)lane * nw < ranks) {
            my_u = a.lo + (uint32_t)(g + (uint64_t)lane * nw);
            const uint64_t W = a.wv[my_u];
            if (W > 1) {  // a bloom takes two wedges
                my_h = a.hv[my_u];
                light = is_light(W, my_h);
            }
        }
        unsigned todo = __ballot_sync(0xffffffffu, light);
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1u;
            const uint32_t u = __shfl_sync(0xffffffffu, my_u, src), h = __shfl_sync(0xffffffffu, my_h, src);
            const uint64_t arc = a.off[u], bb = ea.bloom_base[u], pb = ea.pair_base[u];
            uint32_t len = 0, e = 0;
            uint64_t at = 0;
            if (lane < h) {
                len = a.pl[arc + lane];
                if (len) {
                    e = a.eid[arc + lane];
                    at = a.off[a.adj[arc + lane]];
                }
            }
            const unsigned has = __ballot_sync(0xffffffffu, len > 0u);
            const uint32_t incl = dev::warp_incl_scan(len), total = __shfl_sync(0xffffffffu, incl, 31);
            const uint32_t j = __popc(has & ((1u << lane) - 1u)), n = __popc(has);
            if (len) {
                off[j] = incl - len;
                s_at[wi][j] = at - (incl - len);
                s_e[wi][j] = e | (a.assigned && a.assigned[e] ? 0x80000000u : 0u);
                s_front[wi][j] = ea.inc_off[e];
            }
            if (lane == 31) off[n] = total;
            __syncwarp();
            uint32_t slot[kWin], jj[kWin], j0 = 0;
#pragma unroll
            for (uint32_t r = 0; r < kWin; ++r) {
                slot[r] = kEmpty;
                jj[r] = 0;
                if (32u * r < total) {
                    jj[r] = dev::items_of(off, n, 32u * r, j0);
                    const uint32_t x = 32u * r + lane;
                    if (x < total) slot[r] = a.adj[s_at[wi][jj[r]] + x];
                }
            }
#pragma unroll
            for (uint32_t r = 0; r < kWin; ++r) {
                if (slot[r] == kEmpty) continue;
                const uint32_t w = slot[r];
                uint32_t i = (w * 0x9E3779B1u) >> 23;
                for (;;) {
                    const uint32_t k = atomicCAS(&key[i], kEmpty, w);
                    if (k == kEmpty || k == w) break;
                    i = (i + 1u) & (kSlots - 1u);
                }
                slot[r] = i;
                atomicAdd(&cnt[i], 1u);
            }
            __syncwarp();
            // blooms: cnt becomes the end of the pair range (0: none)
            uint32_t nb = 0, np = 0;
            for (uint32_t i0 = 0; i0 < kSlots; i0 += 32) {
                const uint32_t c = cnt[i0 + lane];
                const bool b = c >= 2u;
                const unsigned m = __ballot_sync(0xffffffffu, b);
                const uint32_t pi = dev::warp_incl_scan(b ? c : 0u);
                if (b) {
                    const uint32_t B = (uint32_t)bb + nb + __popc(m & ((1u << lane) - 1u));
                    const uint32_t end = (uint32_t)pb + np + pi;
                    ea.bloom_k[B] = c;
                    ea.bloom_off[B] = end - c;
                    bloom[i0 + lane] = B;
                    cnt[i0 + lane] = end;
                } else if (c) {
                    cnt[i0 + lane] = 0;
                }
                nb += __popc(m);
                np += __shfl_sync(0xffffffffu, pi, 31);
            }
            __syncwarp();
            // (the pair ranges of a bloom end above 0, and count down within them)
#pragma unroll
            for (uint32_t r = 0; r < kWin; ++r) {
                if (slot[r] == kEmpty || cnt[slot[r]] == 0u) continue;
                const uint32_t p = atomicSub(&cnt[slot[r]], 1u) - 1u, x = 32u * r + lane;
                const uint32_t ev = a.eid[s_at[wi][jj[r]] + x], eu = s_e[wi][jj[r]];
                const bool fu = eu >> 31, fw = a.assigned && a.assigned[ev];
                const unsigned long long back = fw ? 0ull : atomicAdd(&ea.cursor[ev], ~0ull);
                const unsigned long long front = fu ? 0ull : atomicAdd(&s_front[wi][jj[r]], 1ull);
                put_pair(ea, p, bloom[slot[r]], eu & 0x7FFFFFFFu, ev, fu, fw, front, back);
            }
            __syncwarp();
#pragma unroll
            for (uint32_t r = 0; r < kWin; ++r)
                if (slot[r] != kEmpty) {
                    key[slot[r]] = kEmpty;
                    cnt[slot[r]] = 0;
                }
            __syncwarp();
        }
    }
}

}  // namespace

// Whether a kernel whose per-block arrays did not fit the device's memory should be tried
// with half the blocks: they take 4 (count) and 16 bytes (emit) a block for every
// vertex of the larger layer (beyond the counters in shared memory), 460 GB for
// 190M vertices and a block an SM.  A fixed arena has the room it has, and an
// injected failure is one.
static bool fewer_blocks(Alloc &al, unsigned &blocks) {
    if (al.err != cudaErrorMemoryAllocation || al.arena || al.injected || blocks == 1) return false;
    cudaGetLastError();
    al.err = cudaSuccess;
    blocks /= 2;
    return true;
}

cudaError_t count_wedges(const Csr &g, CountOut &o, int num_sms, Alloc &al, uint32_t lo, uint32_t hi) {
    const bool index = o.inc_cnt != nullptr;
    if (hi > g.n) hi = g.n;
    if (lo > hi) lo = hi;
    unsigned blocks = (unsigned)num_sms;
    // ranks below the counters in shared memory (half as many where they have 32
    // bits, for a start vertex of 2^16 middle vertices: its graph has those and more)
    const uint32_t width = g.cnt_n < 0x10000u ? kHot : kHot / 2;
    CountArgs a{};
    a.off = g.off;
    a.adj = g.adj;
    a.place = g.place;
    a.wend = g.place ? g.wplace : g.adj;
    a.eid = g.eid;
    a.hv = g.hv;
    a.pl = g.pl;
    a.wv = g.wv;
    a.heavy = g.heavy;
    a.n_heavy = g.n_heavy;
    a.lo = lo;
    a.hi = hi;
    a.vbase = g.vbase;
    a.cold_n = g.cnt_n > width ? g.cnt_n - width : 0u;
    a.queue = al.get<uint32_t>(1);
    if (al.err != cudaSuccess) return al.err;
    while (!(a.cold = al.get<uint32_t>((size_t)blocks * a.cold_n)) && fewer_blocks(al, blocks)) {
    }
    a.totals = reinterpret_cast<unsigned long long *>(g.totals + 1);
    if (al.err != cudaSuccess) return al.err;
    a.support = reinterpret_cast<unsigned long long *>(o.support);
    a.inc_cnt = o.inc_cnt;
    a.w2v = o.w2v;
    a.nbv = o.nbv;
    a.assigned = index ? o.assigned : nullptr;
    if (a.cold_n) BT_CUDA(cudaMemsetAsync(a.cold, 0, sizeof(uint32_t) * (size_t)blocks * a.cold_n, al.stream));
    BT_CUDA(cudaMemsetAsync(a.queue, 0, sizeof(uint32_t), al.stream));
    BT_CUDA(cudaMemsetAsync(o.support, 0, sizeof(uint64_t) * g.m, al.stream));
    if (index) BT_CUDA(cudaMemsetAsync(o.inc_cnt, 0, sizeof(uint32_t) * g.m, al.stream));
    const size_t smem = sizeof(CountShared) + kHot * sizeof(uint16_t);
    const unsigned groups = (hi - lo + 7u) / 8u, room = (unsigned)num_sms * 5u;
    const unsigned light = groups < room ? (groups ? groups : 1u) : room;
    al.mark(kPhCount, false);
    if (index) {
        BT_CUDA(cudaFuncSetAttribute(k_count<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        k_count<true><<<blocks, kCT, smem, al.stream>>>(a);
        k_count_light<true><<<light, 256, 0, al.stream>>>(a);
    } else {
        BT_CUDA(cudaFuncSetAttribute(k_count<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        k_count<false><<<blocks, kCT, smem, al.stream>>>(a);
        k_count_light<false><<<light, 256, 0, al.stream>>>(a);
    }
    al.launches += 2;
    al.mark(kPhCount, true);
    BT_CUDA(cudaGetLastError());
    al.put(a.cold);
    al.put(a.queue);
    return cudaSuccess;
}

cudaError_t emit_index(const Csr &g, const CountOut &c, Index &ix, int num_sms, Alloc &al, cudaStream_t stream) {
    const uint32_t n = g.n;
    const uint64_t m = g.m;
    ix.m = m;
    // layout prefix sums
    uint64_t *bloom_base = al.get<uint64_t>(n);
    uint64_t *pair_base = al.get<uint64_t>(n);
    uint64_t *tot = g.totals + 2;
    uint64_t *incc64 = al.get<uint64_t>(m + 1);
    ix.inc_off = al.get<uint64_t>(m + 1);
    if (al.err != cudaSuccess) return al.err;
    BT_CUDA(exclusive_scan_u64(c.nbv, bloom_base, n, tot + 0, al));
    BT_CUDA(exclusive_scan_u64(c.w2v, pair_base, n, tot + 1, al));
    BT_CUDA(widen_u32(c.inc_cnt, incc64, m, al));
    BT_CUDA(cudaMemsetAsync(incc64 + m, 0, sizeof(uint64_t), al.stream));
    BT_CUDA(exclusive_scan_u64(incc64, ix.inc_off, m + 1, tot + 2, al));
    uint64_t h_tot[5];
    BT_CUDA(cudaMemcpyAsync(h_tot, g.totals, sizeof(h_tot), cudaMemcpyDeviceToHost, stream));
    BT_CUDA(cudaStreamSynchronize(stream));
    ix.w = h_tot[0];
    ix.butterflies = h_tot[1] / 2;  // every butterfly gives each of its two wedges in a bloom one
    ix.nb = h_tot[2];
    ix.w2 = h_tot[3];
    ix.links = h_tot[4];  // 2 w2, less the links of assigned edges in a compressed index
    // pair ids are u32; bloom ids keep bit 31 free for the link's side
    if (ix.w2 >= 0xFFFFFFFFull || ix.nb >= 0x80000000ull) {
        al.put(bloom_base);
        al.put(pair_base);
        al.put(incc64);
        return cudaErrorInvalidValue;  // reported as overflow by the caller
    }
    ix.bloom_k = al.get<uint32_t>(ix.nb);
    ix.bloom_off = al.get<uint32_t>(ix.nb + 1);
    ix.pairs = al.get<uint2>(ix.w2);
    ix.inc = al.get<uint2>(ix.links);
    unsigned blocks = (unsigned)num_sms;
    EmitArgs a{};
    a.c.off = g.off;
    a.c.adj = g.adj;
    a.c.place = g.place;
    a.c.wend = g.place ? g.wplace : g.adj;
    a.c.eid = g.eid;
    a.c.hv = g.hv;
    a.c.pl = g.pl;
    a.c.wv = g.wv;
    a.c.hi = n;
    a.c.heavy = g.heavy;
    a.c.n_heavy = g.n_heavy;
    a.c.vbase = g.vbase;
    const uint32_t width = g.cnt_n < 0x10000u ? kHotE : kHotE / 2;  // as in count_wedges
    a.c.cold_n = g.cnt_n > width ? g.cnt_n - width : 0u;
    a.c.queue = al.get<uint32_t>(1);
    a.c.assigned = c.assigned;
    if (al.err != cudaSuccess) return al.err;
    for (;;) {
        const size_t held = al.live.size();
        a.c.cold = al.get<uint32_t>((size_t)blocks * a.c.cold_n);
        a.word = al.get<unsigned long long>((size_t)blocks * g.cnt_n);
        a.found = al.get<uint32_t>((size_t)blocks * a.c.cold_n);
        if (al.err == cudaSuccess) break;
        if (!fewer_blocks(al, blocks)) return al.err;
        al.undo_to(held);
        BT_CUDA(cudaStreamSynchronize(stream));
    }
    a.cnt_n = g.cnt_n;
    a.bloom_base = bloom_base;
    a.pair_base = pair_base;
    a.inc_off = ix.inc_off;
    a.cursor = reinterpret_cast<unsigned long long *>(incc64);
    a.bloom_k = ix.bloom_k;
    a.bloom_off = ix.bloom_off;
    a.pairs = ix.pairs;
    a.inc = ix.inc;
    a.twin = ix.twin_links;
    uint32_t w2_32 = (uint32_t)ix.w2;
    BT_CUDA(cudaMemcpyAsync(ix.bloom_off + ix.nb, &w2_32, sizeof(uint32_t), cudaMemcpyHostToDevice,
                            stream));
    // the lists are filled from their ends too
    BT_CUDA(cudaMemcpyAsync(a.cursor, ix.inc_off + 1, sizeof(uint64_t) * m, cudaMemcpyDeviceToDevice, al.stream));
    if (a.c.cold_n) BT_CUDA(cudaMemsetAsync(a.c.cold, 0, sizeof(uint32_t) * (size_t)blocks * a.c.cold_n, al.stream));
    BT_CUDA(cudaMemsetAsync(a.c.queue, 0, sizeof(uint32_t), al.stream));
    const size_t smem = sizeof(EmitShared) + kHotE * sizeof(uint16_t);
    const unsigned groups = (n + 7u) / 8u, room = (unsigned)num_sms * 4u;
    al.mark(kPhEmit, false);
    BT_CUDA(cudaFuncSetAttribute(k_emit, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_emit<<<blocks, kCT, smem, al.stream>>>(a);
    k_emit_light<<<groups < room ? (groups ? groups : 1u) : room, 256, 0, al.stream>>>(a);
    al.launches += 2;
    al.mark(kPhEmit, true);
    BT_CUDA(cudaGetLastError());
    // the host copy of w2_32 must outlive the async copy
    BT_CUDA(cudaStreamSynchronize(stream));
    al.put(a.c.cold);
    al.put(a.c.queue);
    al.put(a.word);
    al.put(a.found);
    al.put(incc64);
    al.put(bloom_base);
    al.put(pair_base);
    return cudaSuccess;
}

namespace {
__device__ __forceinline__ uint32_t first_at_least(const uint64_t *pre, uint32_t n, uint64_t t) {
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
        const uint32_t mid = lo + (hi - lo) / 2;
        if (pre[mid] < t) lo = mid + 1; else hi = mid;
    }
    return lo;
}
__global__ void k_rank_bounds(const uint64_t *pre, uint32_t n, uint64_t t0, uint64_t t1, uint32_t *out) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        out[0] = first_at_least(pre, n, t0);
        out[1] = first_at_least(pre, n, t1);
    }
}
}  // namespace

cudaError_t rank_bounds(const uint64_t *pre, uint32_t n, uint64_t t0, uint64_t t1, uint32_t *out, Alloc &al) {
    k_rank_bounds<<<1, 32, 0, al.stream>>>(pre, n, t0, t1, out);
    al.launches++;
    return cudaGetLastError();
}

void free_index(Index &ix, Alloc &al) {
    al.put(ix.newid);
    al.put(ix.bloom_k);
    al.put(ix.bloom_off);
    al.put(ix.pairs);
    al.put(ix.inc_off);
    al.put(ix.inc);
    ix = Index{};
}

}  // namespace bt
