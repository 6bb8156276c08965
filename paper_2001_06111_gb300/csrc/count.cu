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
// ranks just below the start vertex, the ones most wedges end at, are in shared
// memory, and only those of lower ranks are in global memory.
// Emit: persistent blocks pull start vertices from a queue, walk their wedges in
// chunks of NT middle vertices (NT = block size, picked by the batch autotuner
// from 256, 512, 1024), with a dense array of 64-bit words a block (count and
// claimed bloom) indexed by rank, kept at zero between vertices.
#include "bt_device.cuh"
#include "bt_internal.cuh"

namespace bt {
namespace {

template <int NT>
struct Chunk {
    uint32_t off[NT + 1];  // exclusive prefix of wedge counts; off[NT] = total
    uint32_t v[NT];        // middle vertex (rank)
    uint32_t e[NT];        // edge id of (u, v)
};

// Loads middle vertices [c0, c0 + NT) of start vertex u.  Returns the
// number of wedges in the chunk.  Contains __syncthreads().
template <int NT>
__device__ __forceinline__ uint32_t load_chunk(Chunk<NT> &ch, const uint32_t *adj, const uint32_t *eid,
                                               const uint32_t *pl, uint64_t a, uint32_t h,
                                               uint32_t c0) {
    uint32_t i = c0 + threadIdx.x;
    uint32_t p = 0, v = 0, e = 0;
    if (i < h) {
        p = pl[a + i];
        v = adj[a + i];
        e = eid[a + i];
    }
    uint32_t tot;
    uint32_t ex = dev::block_excl_scan<uint32_t>(p, &tot);
    ch.off[threadIdx.x] = ex;
    ch.v[threadIdx.x] = v;
    ch.e[threadIdx.x] = e;
    if (threadIdx.x == 0) ch.off[NT] = tot;
    __syncthreads();
    return tot;
}

// Wedge t of the chunk -> (chunk slot vi, arc index of (v, w) in the CSR).
template <int NT>
__device__ __forceinline__ uint64_t wedge_arc(const Chunk<NT> &ch, const uint64_t *off, uint32_t t,
                                              uint32_t &vi) {
    vi = dev::last_le_u32(ch.off, NT, t);
    return off[ch.v[vi]] + (t - ch.off[vi]);
}

// Next start vertex of the rank range [lo, hi), highest rank first.
__device__ __forceinline__ uint32_t next_vertex(uint32_t *queue, uint32_t lo, uint32_t hi, uint32_t *s_q) {
    if (threadIdx.x == 0) *s_q = atomicAdd(queue, 1u);
    __syncthreads();
    uint32_t qi = *s_q;
    __syncthreads();
    return qi < hi - lo ? hi - 1 - qi : 0xFFFFFFFFu;
}

__device__ __forceinline__ uint32_t ld_cg(const uint32_t *p) { return __ldcg(p); }

// Pass A on emit's packed words (count in the low 32 bits).
template <int NT>
__device__ void pass_count64(Chunk<NT> &ch, const uint64_t *off, const uint32_t *adj,
                             const uint32_t *eid, const uint32_t *pl, uint64_t a, uint32_t h,
                             unsigned long long *cw, uint32_t vb) {
    for (uint32_t c0 = 0; c0 < h; c0 += NT) {
        uint32_t T = load_chunk(ch, adj, eid, pl, a, h, c0);
        for (uint32_t t = threadIdx.x; t < T; t += NT) {
            uint32_t vi;
            uint64_t arc = wedge_arc(ch, off, t, vi);
            atomicAdd(&cw[adj[arc] - vb], 1ull);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------- count
constexpr int kCT = 1024;                // threads of a count block (one an SM)
constexpr uint32_t kCU = 4;              // wedges a lane has in flight
constexpr uint32_t kHot = 88 * 1024;     // 16-bit counters in shared memory

struct CountArgs {
    const uint64_t *off;
    const uint32_t *adj, *eid, *hv, *pl;
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
    uint32_t acc[kCT], inc[kCT];     // support and links of (u, v) from these (supports are below m < 2^31)
    uint32_t u;
};

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
// of the kHot ranks below u are in shared memory (ranks ascend with degree, so
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
    const uint32_t n_heavy = *a.n_heavy;
    if (tid == 0) s.u = atomicAdd(a.queue, 1u);
    __syncthreads();
    for (;;) {
        const uint32_t q = s.u;
        if (q >= n_heavy) break;
        __syncthreads();
        uint32_t next = 0;  // the following turn, asked for ahead
        if (tid == 0) next = atomicAdd(a.queue, 1u);
        const uint32_t u = a.heavy[n_heavy - 1u - q];
        if (u >= a.lo && u < a.hi) {
            const uint64_t arc = a.off[u];
            const uint32_t h = a.hv[u];
            const uint32_t vb = a.vbase ? a.vbase[u] : 0u;
            const bool narrow = h < 0x10000u;  // a count never exceeds h
            const uint32_t width = narrow ? kHot : kHot / 2;
            const uint32_t ru = u - vb;
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
                        w[r] = x < hi ? a.adj[s.at[j] + x] - vb : 0xFFFFFFFFu;
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
                        w[r] = x < hi ? a.adj[s.at[jj[r]] + x] - vb : 0xFFFFFFFFu;
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
                        const uint32_t w = x < hi ? a.adj[s.at[j] + x] - vb : 0xFFFFFFFFu;
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

// Emit the index: blooms (bloom number, first pair), twin pairs and the
// per-edge link lists.  The dense per-block array holds one 64-bit word per
// end vertex: the wedge count in the low half and, once the bloom is claimed,
// 2 + its index among the vertex's blooms in the high half, so a wedge reads
// and updates one word (one memory sector) in every pass.
template <int NT>
__global__ void __launch_bounds__(NT) k_emit(
    const uint64_t *__restrict__ off, const uint32_t *__restrict__ adj,
    const uint32_t *__restrict__ eid, const uint32_t *__restrict__ hv,
    const uint32_t *__restrict__ pl, const uint64_t *__restrict__ wv, uint32_t n,
    const uint32_t *__restrict__ vbase, uint32_t cn,
    unsigned long long *cw_all, const uint64_t *__restrict__ bloom_base,
    const uint64_t *__restrict__ pair_base, const uint64_t *__restrict__ inc_off,
    uint32_t *inc_fill, uint32_t *bloom_k, uint32_t *bloom_off, uint2 *pairs,
    uint2 *inc, uint32_t *queue, const uint8_t *__restrict__ assigned, bool twin) {
    __shared__ Chunk<NT> ch;
    __shared__ uint32_t s_q;
    // bloom count (high 32 bits) and pair count (low 32 bits) of the vertex,
    // advanced by one atomic so that pair ranges follow bloom ids
    __shared__ unsigned long long s_alloc;
    unsigned long long *cw = cw_all + (size_t)blockIdx.x * cn;
    for (;;) {
        uint32_t u = next_vertex(queue, 0u, n, &s_q);
        if (u == 0xFFFFFFFFu) break;
        if (wv[u] == 0) continue;
        const uint64_t a = off[u];
        const uint32_t h = hv[u];
        const uint64_t bb = bloom_base[u];
        const uint64_t pb = pair_base[u];
        const uint32_t vb = vbase ? vbase[u] : 0u;
        if (threadIdx.x == 0) s_alloc = 0;
        pass_count64(ch, off, adj, eid, pl, a, h, cw, vb);
        // claim: one thread per bloom allocates its id and pair range
        for (uint32_t c0 = 0; c0 < h; c0 += NT) {
            uint32_t T = load_chunk(ch, adj, eid, pl, a, h, c0);
            for (uint32_t t = threadIdx.x; t < T; t += NT) {
                uint32_t vi;
                uint64_t arc = wedge_arc(ch, off, t, vi);
                const uint32_t w = adj[arc] - vb;  // counter index
                const unsigned long long x = __ldcg(&cw[w]);
                const uint32_t c = (uint32_t)x;
                // a single wedge is the only reader of its word: clear it now
                if (c == 1u) cw[w] = 0ull;
                if (c >= 2 && atomicCAS(&cw[w], (unsigned long long)c, 1ull << 32 | c) == (unsigned long long)c) {
                    unsigned long long old = atomicAdd(&s_alloc, (1ull << 32) | c);
                    uint32_t j = (uint32_t)(old >> 32);
                    uint32_t p = (uint32_t)old;
                    uint64_t B = bb + j;
                    bloom_k[B] = c;
                    bloom_off[B] = (uint32_t)(pb + p);
                    atomicExch(&cw[w], (unsigned long long)(j + 2u) << 32 | c);
                }
            }
            __syncthreads();
        }
        // place each bloom wedge as a twin pair and link both edges to it
        for (uint32_t c0 = 0; c0 < h; c0 += NT) {
            uint32_t T = load_chunk(ch, adj, eid, pl, a, h, c0);
            for (uint32_t t = threadIdx.x; t < T; t += NT) {
                uint32_t vi;
                uint64_t arc = wedge_arc(ch, off, t, vi);
                const uint32_t w = adj[arc] - vb;  // counter index
                const uint32_t x = (uint32_t)(__ldcg(&cw[w]) >> 32);
                if (x >= 2) {
                    uint64_t B = bb + (x - 2);
                    // the low half counts down the bloom's wedges still to place
                    uint32_t pos = (uint32_t)atomicAdd(&cw[w], ~0ull) - 1u;
                    // the last wedge of the bloom comes after every read of the
                    // word (each precedes its own decrement): clear it
                    if (pos == 0u) cw[w] = 0ull;
                    uint32_t slot = ld_cg(&bloom_off[B]) + pos;
                    uint32_t euv = ch.e[vi], evw = eid[arc];
                    const bool fu = assigned && assigned[euv], fw = assigned && assigned[evw];
                    // an assigned edge is flagged in bit 31 and gets no link
                    pairs[slot] = make_uint2(euv | (fu ? 0x80000000u : 0u), evw | (fw ? 0x80000000u : 0u));
                    // each link carries its bloom and which member of the pair
                    // the edge is, or the twin itself and the bloom
                    if (!fu) {
                        uint32_t q1 = atomicAdd(&inc_fill[euv], 1u);
                        inc[inc_off[euv] + q1] = make_uint2(twin ? evw : slot, (uint32_t)B);
                    }
                    if (!fw) {
                        uint32_t q2 = atomicAdd(&inc_fill[evw], 1u);
                        inc[inc_off[evw] + q2] = make_uint2(twin ? euv : slot, (uint32_t)B | (twin ? 0u : 0x80000000u));
                    }
                }
            }
            __syncthreads();
        }
    }
}

}  // namespace

cudaError_t count_wedges(const Csr &g, CountOut &o, int num_sms, Alloc &al, uint32_t lo, uint32_t hi) {
    const bool index = o.inc_cnt != nullptr;
    if (hi > g.n) hi = g.n;
    if (lo > hi) lo = hi;
    const unsigned blocks = (unsigned)num_sms;
    // ranks below the counters in shared memory (half as many where they have 32
    // bits, for a start vertex of 2^16 middle vertices: its graph has those and more)
    const uint32_t width = g.cnt_n < 0x10000u ? kHot : kHot / 2;
    CountArgs a{};
    a.off = g.off;
    a.adj = g.adj;
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
    a.cold = al.get<uint32_t>((size_t)blocks * a.cold_n);
    a.queue = al.get<uint32_t>(1);
    a.totals = al.get<unsigned long long>(1);
    if (al.err != cudaSuccess) return al.err;
    a.support = reinterpret_cast<unsigned long long *>(o.support);
    a.inc_cnt = o.inc_cnt;
    a.w2v = o.w2v;
    a.nbv = o.nbv;
    a.assigned = index ? o.assigned : nullptr;
    if (a.cold_n) BT_CUDA(cudaMemsetAsync(a.cold, 0, sizeof(uint32_t) * (size_t)blocks * a.cold_n, al.stream));
    BT_CUDA(cudaMemsetAsync(a.queue, 0, sizeof(uint32_t), al.stream));
    BT_CUDA(cudaMemsetAsync(a.totals, 0, sizeof(unsigned long long), al.stream));
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
    o.butterflies_dev = a.totals;
    al.put(a.cold);
    al.put(a.queue);
    return cudaSuccess;
}

cudaError_t emit_index(const Csr &g, const CountOut &c, Index &ix, int num_sms, Alloc &al,
                       cudaStream_t stream, int nt) {
    if (nt != 256 && nt != 1024) nt = 512;
    const uint32_t n = g.n;
    const uint64_t m = g.m;
    ix.m = m;
    // layout prefix sums
    uint64_t *bloom_base = al.get<uint64_t>(n);
    uint64_t *pair_base = al.get<uint64_t>(n);
    uint64_t *tot = al.get<uint64_t>(3);
    uint64_t *incc64 = al.get<uint64_t>(m + 1);
    ix.inc_off = al.get<uint64_t>(m + 1);
    if (al.err != cudaSuccess) return al.err;
    BT_CUDA(exclusive_scan_u64(c.nbv, bloom_base, n, tot + 0, al));
    BT_CUDA(exclusive_scan_u64(c.w2v, pair_base, n, tot + 1, al));
    BT_CUDA(widen_u32(c.inc_cnt, incc64, m, al));
    BT_CUDA(cudaMemsetAsync(incc64 + m, 0, sizeof(uint64_t), al.stream));
    BT_CUDA(exclusive_scan_u64(incc64, ix.inc_off, m + 1, tot + 2, al));
    al.put(incc64);
    uint64_t h_tot[3];
    BT_CUDA(cudaMemcpyAsync(h_tot, tot, sizeof(h_tot), cudaMemcpyDeviceToHost, stream));
    BT_CUDA(cudaStreamSynchronize(stream));
    ix.nb = h_tot[0];
    ix.w2 = h_tot[1];
    ix.links = h_tot[2];  // 2 w2, less the links of assigned edges in a compressed index
    // pair ids are u32; bloom ids keep bit 31 free for the link's side
    if (ix.w2 >= 0xFFFFFFFFull || ix.nb >= 0x80000000ull) {
        al.put(bloom_base);
        al.put(pair_base);
        al.put(tot);
        return cudaErrorInvalidValue;  // reported as overflow by the caller
    }
    ix.bloom_k = al.get<uint32_t>(ix.nb);
    ix.bloom_off = al.get<uint32_t>(ix.nb + 1);
    ix.pairs = al.get<uint2>(ix.w2);
    ix.inc = al.get<uint2>(ix.links);
    uint32_t *inc_fill = al.get<uint32_t>(m);
    // as few resident blocks as keep the SMs busy, so that few of their dense
    // arrays compete for L2 (1024 threads: one block an SM measured 5-20 % faster
    // than two; a batch of 384 graphs with 256 threads: 8.7 ms with six, 10.0 with eight)
    const int bps = nt == 1024 ? 1 : nt == 512 ? 3 : 6;
    unsigned blocks = (unsigned)(num_sms * bps);
    unsigned long long *cw = al.get<unsigned long long>((size_t)blocks * g.cnt_n);
    uint32_t *queue = al.get<uint32_t>(1);
    if (al.err != cudaSuccess) return al.err;
    uint32_t w2_32 = (uint32_t)ix.w2;
    BT_CUDA(cudaMemcpyAsync(ix.bloom_off + ix.nb, &w2_32, sizeof(uint32_t), cudaMemcpyHostToDevice,
                            stream));
    BT_CUDA(cudaMemsetAsync(inc_fill, 0, sizeof(uint32_t) * m, al.stream));
    BT_CUDA(cudaMemsetAsync(cw, 0, sizeof(unsigned long long) * (size_t)blocks * g.cnt_n, al.stream));
    BT_CUDA(cudaMemsetAsync(queue, 0, sizeof(uint32_t), al.stream));
    al.mark(kPhEmit, false);
#define BT_EMIT_ARGS                                                                         \
    g.off, g.adj, g.eid, g.hv, g.pl, g.wv, n, g.vbase, g.cnt_n, cw, bloom_base, pair_base, ix.inc_off,  \
        inc_fill, ix.bloom_k, ix.bloom_off, ix.pairs, ix.inc, queue, c.assigned, ix.twin_links
    if (nt == 256) k_emit<256><<<blocks, 256, 0, al.stream>>>(BT_EMIT_ARGS);
    else if (nt == 1024) k_emit<1024><<<blocks, 1024, 0, al.stream>>>(BT_EMIT_ARGS);
    else k_emit<512><<<blocks, 512, 0, al.stream>>>(BT_EMIT_ARGS);
#undef BT_EMIT_ARGS
    al.launches++;
    al.mark(kPhEmit, true);
    BT_CUDA(cudaGetLastError());
    // the host copy of w2_32 must outlive the async copy
    BT_CUDA(cudaStreamSynchronize(stream));
    al.put(cw);
    al.put(queue);
    al.put(inc_fill);
    al.put(bloom_base);
    al.put(pair_base);
    al.put(tot);
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
