// Part graphs for the part peel (local.cu): a whole small graph, or the ranges of
// bitruss numbers a coarse peel found.
//
// Ranges.  The coarse peel (peel.cu) gives every edge the part its bitruss
// number falls in, parts ascending.  When part q begins, all edges of lower
// parts are gone, so of a bloom's twin pairs those with both edges in parts >= q
// remain; Alg. 5 inside part q then needs
//   * the bloom number k_B at that point: the pairs whose lower edge is in a
//     part >= q;
//   * the pairs that can die inside part q: those whose lower edge is in q.  An
//     edge of a higher part is flagged: it is not peeled here and its support
//     is not updated.
// A pair thus belongs to one part, min(part(e1), part(e2)), and a bloom falls
// apart into one group of pairs a part.  A group whose k_B is 1 holds no
// butterfly and is dropped.  Supports at the start of a part come from the
// coarse peel, so each part is peeled without any other.
#include <algorithm>
#include <cmath>
#include <vector>

#include "bt_device.cuh"
#include "bt_internal.cuh"

namespace bt {
namespace {

constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr uint32_t kFlag = 0x80000000u;
constexpr uint32_t kMaxParts = kPartsMax;
constexpr int kT = 256;
// A part with more links than this many times the mean is peeled by a cluster.  Peel
// with 2.5 instead: 200,000 edges 8.9 against 7.4 ms, 2M edges 74.2 against 69.0
// (the clusters take the SMs of the other parts, and their barriers cost more);
// with 6 or 12: the same within 1 %.
constexpr double kHeavy = 4.0;
// The mean says nothing where there are few parts: with fewer than kFewParts the
// limit is that of as many, but at least kBlockLinks links, 1 to 2 ms of one
// block (K_{200,200} of 8M links beside smaller bicliques: 10 ms by one block).
constexpr double kFewParts = 40.0;
constexpr double kBlockLinks = 1 << 19;
// What a part takes by itself, nanoseconds a link by a block (2.9 to 5.1: random
// graphs of 20,000 edges, blocks of 100 x 100) and a link and an edge by a cluster
// (0.37 to 0.57: random graphs of 1M and 2M edges, a block of 1000 x 1000; 4.3:
// edges in no butterfly).  The grid takes 8 us for each round of every part in turn, 2
// more than a block, and 0.1 ns a link.  Rounds of a part on skewed graphs: 57 at
// 5,000 links, 82 at 24,000, 165 at 114,000, 471 at 1.2M, and no more than 600.  Where
// the longest part takes longer than all that, the rounds of a first part that
// would be made again among it, it is no range among others: the grid peels the graph.  (Three random graphs of 0.5M to 2M edges by
// parts 157 ms, by the grid 122; two sizes of bicliques 13.4 and 1.8; a 300 x 300 block in
// a skewed graph of 200,000 edges 15.4 and 32.)
constexpr double kBlockLinkNs = 3.7, kClusterLinkNs = 0.45, kClusterEdgeNs = 4.3;
constexpr double kGridRoundNs = 8000.0, kGridMoreNs = 2000.0, kGridLinkNs = 0.1;
inline double rounds_of(double links) { return std::min(600.0, 57.0 * std::pow(links / 5000.0, 0.45)); }
constexpr int kSmall = 8;  // pairs of a bloom that one thread groups by itself
constexpr unsigned kFull = 0xffffffffu;

inline unsigned grid_for(uint64_t items, int threads, unsigned cap) {
    uint64_t g = (items + threads - 1) / threads;
    if (g == 0) g = 1;
    return (unsigned)(g < cap ? g : cap);
}

__device__ __forceinline__ void head(BloomRec *b, uint32_t first, uint32_t n, uint32_t k) {
    *reinterpret_cast<uint4 *>(b) = make_uint4(first, n, k, 0u);
}

__global__ void k_bloom_rec(const uint32_t *bloom_k, const uint32_t *bloom_off, const uint2 *pairs, uint64_t nb,
                            BloomRec *bl) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < nb; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t o = bloom_off[i], n = bloom_off[i + 1] - o;
        head(bl + i, o, n, bloom_k[i]);
        if (n <= 2u)
            for (uint32_t j = 0; j < n; ++j) bl[i].pair[j] = pairs[o + j];
    }
}

// Edge records of the whole graph; ends: its first and last edge, first and last bloom.
__global__ void k_edge_rec(const uint64_t *inc_off, const uint64_t *support, uint64_t m, uint32_t nb, uint32_t *ends,
                           uint4 *er) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<uint4 *>(ends) = make_uint4(0u, (uint32_t)m, 0u, nb);
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t o = inc_off[i];
        er[i] = make_uint4((uint32_t)o, (uint32_t)(o >> 32), (uint32_t)(inc_off[i + 1] - o), (uint32_t)support[i]);
    }
}

// Sort keys: the part of an edge, np for an assigned one.
__global__ void k_iota2(const uint32_t *part, const uint8_t *assigned, uint32_t np, uint64_t m, uint32_t *keys,
                        uint32_t *vals) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x) {
        keys[i] = assigned && assigned[i] ? np : part[i];
        vals[i] = (uint32_t)i;
    }
}

// keys: parts in ascending order (np of them; np: assigned), order: the edges.
// place[e] = (new id, part); part_e[q]: the first edge of part q.
__global__ void k_place(const uint32_t *keys, const uint32_t *order, uint64_t m, uint32_t np, uint2 *place,
                        uint32_t *part_e) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t q = keys[i];
        place[order[i]] = make_uint2(q < np ? (uint32_t)i : kAssigned, q);
        const uint32_t before = i ? keys[i - 1] + 1u : 0u;  // a part may be empty
        for (uint32_t x = before; x <= q; ++x) part_e[x] = (uint32_t)i;
        if (i + 1 == m)
            for (uint32_t x = q + 1u; x <= np; ++x) part_e[x] = (uint32_t)m;
    }
}

struct SplitArgs {
    const uint32_t *bloom_off;
    uint64_t nb;
    const uint2 *pairs;   // the index's
    const uint2 *place;   // per edge: new id, part
    uint32_t np;
    uint2 *out;           // pairs of groups of more than two, part by part, new ids
    uint32_t *sub;        // per pair of the index: its group, or kNone
    BloomRec *bl;         // group records, part by part
    uint32_t *groups;     // [np] groups of each part: counted, then (the exclusive sums) handed out
    uint32_t *members;    // [np] their pairs (of groups of more than two), likewise
    bool assigned;        // some edges are assigned (part np): flagged in the index's pairs
};

__device__ __forceinline__ uint2 placed(uint2 a, uint2 b) {
    return make_uint2(a.x | (a.y > b.y ? kFlag : 0u), b.x | (b.y > a.y ? kFlag : 0u));
}

// What a block takes of each part's groups and pairs: counted in shared memory,
// then added to the part's counters with one atomic a part.
struct Tally {
    uint32_t groups[kMaxParts], members[kMaxParts];
};
__device__ __forceinline__ void tally_zero(Tally &s, uint32_t np) {
    for (uint32_t i = threadIdx.x; i < np; i += kT) s.groups[i] = s.members[i] = 0;
}
// s becomes the first of the places taken (kTake), or is only added.
template <bool kTake>
__device__ __forceinline__ void tally_add(Tally &s, const SplitArgs &a) {
    for (uint32_t i = threadIdx.x; i < a.np; i += kT) {
        const uint32_t g = s.groups[i], n = s.members[i];
        if (!g) continue;
        const uint32_t g0 = atomicAdd(&a.groups[i], g), n0 = n ? atomicAdd(&a.members[i], n) : 0u;
        if (kTake) {
            s.groups[i] = g0;
            s.members[i] = n0;
        }
    }
}

// Blooms of up to kSmall pairs, one thread each, all its pairs in registers.
// kPlace: places the groups; else counts them.
template <bool kPlace>
__global__ void __launch_bounds__(kT) k_split_small(const SplitArgs a) {
    __shared__ Tally s;
    tally_zero(s, a.np);
    __syncthreads();
    for (uint64_t b0 = (uint64_t)blockIdx.x * kT; b0 < a.nb; b0 += (uint64_t)gridDim.x * kT) {
        const uint64_t B = b0 + threadIdx.x;
        uint32_t off = 0, K = 0;
        if (B < a.nb) {
            off = a.bloom_off[B];
            K = a.bloom_off[B + 1] - off;
            if (K > (uint32_t)kSmall) K = 0;
        }
        uint2 px[kSmall], py[kSmall];
        uint32_t q[kSmall];
#pragma unroll
        for (int i = 0; i < kSmall; ++i) px[i] = (uint32_t)i < K ? a.pairs[off + i] : make_uint2(0u, 0u);
#pragma unroll
        for (int i = 0; i < kSmall; ++i) {
            const uint2 pr = px[i];
            py[i] = (uint32_t)i < K ? a.place[pr.y & ~kFlag] : make_uint2(0u, 0u);
            px[i] = (uint32_t)i < K ? a.place[pr.x & ~kFlag] : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int i = 0; i < kSmall; ++i) q[i] = (uint32_t)i < K ? (px[i].y < py[i].y ? px[i].y : py[i].y) : kNone;
        // size and first pair of every pair's group; left: its k_B
        uint32_t left[kSmall], rank[kSmall], first[kSmall], size[kSmall];
#pragma unroll
        for (int i = 0; i < kSmall; ++i) {
            left[i] = K;
            rank[i] = size[i] = 0;
            first[i] = i;
#pragma unroll
            for (int j = kSmall - 1; j >= 0; --j) {
                left[i] -= q[j] < q[i];
                rank[i] += j < i && q[j] == q[i];
                size[i] += q[j] == q[i];
                if (q[j] == q[i]) first[i] = j;
            }
            if ((uint32_t)i < K && first[i] == (uint32_t)i && left[i] >= 2u && q[i] < a.np) {
                atomicAdd(&s.groups[q[i]], 1u);
                if (size[i] > 2u) atomicAdd(&s.members[q[i]], size[i]);
            }
        }
        if constexpr (kPlace) {
            __syncthreads();
            tally_add<true>(s, a);
            __syncthreads();
            uint32_t id[kSmall], at[kSmall];
#pragma unroll
            for (int i = 0; i < kSmall; ++i) {
                id[i] = kNone;
                at[i] = 0;
                if ((uint32_t)i < K && first[i] == (uint32_t)i && left[i] >= 2u && q[i] < a.np) {
                    id[i] = atomicAdd(&s.groups[q[i]], 1u);
                    if (size[i] > 2u) at[i] = atomicAdd(&s.members[q[i]], size[i]);
                    uint32_t known = 0;  // assigned edges among the pairs of higher parts
                    if (a.assigned)
#pragma unroll
                        for (int j = 0; j < kSmall; ++j)
                            if ((uint32_t)j < K && q[j] > q[i]) known += (px[j].y == a.np) + (py[j].y == a.np);
                    head(a.bl + id[i], size[i] > 2u ? at[i] : known, size[i], left[i]);
                    if (size[i] > 2u) a.bl[id[i]].pair[0].x = known;
                }
#pragma unroll
                for (int j = 0; j < i; ++j)
                    if (first[i] == (uint32_t)j) {
                        id[i] = id[j];
                        at[i] = at[j];
                    }
                if ((uint32_t)i < K) {
                    a.sub[off + i] = id[i];
                    if (id[i] != kNone) {
                        uint2 *to = size[i] > 2u ? a.out + at[i] : a.bl[id[i]].pair;
                        to[rank[i]] = placed(px[i], py[i]);
                    }
                }
            }
            __syncthreads();
            tally_zero(s, a.np);
            __syncthreads();
        }
    }
    if constexpr (!kPlace) {
        __syncthreads();
        tally_add<false>(s, a);
    }
}

// Larger blooms, one warp each: a histogram over the parts in shared memory.
template <bool kPlace>
__global__ void __launch_bounds__(kT) k_split_large(const SplitArgs a) {
    constexpr int kWarps = kT / 32;
    extern __shared__ uint32_t s_tab[];  // three rows a warp; then the block's tally
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t row = a.np + 1u;
    // a part's pairs, then the next place of its group's; its group; its assigned
    // edges, then the size of its group (places take all 32 bits, so what tells a
    // group in the record from one in `out` is a row of its own)
    uint32_t *cur = s_tab + (size_t)w * 3 * row, *gid = cur + row, *known = gid + row, *size = known;
    uint32_t *t_groups = s_tab + (size_t)kWarps * 3 * row, *t_members = t_groups + row;
    if constexpr (!kPlace) {
        for (uint32_t i = threadIdx.x; i < 2 * row; i += kT) t_groups[i] = 0;
        __syncthreads();
    }
    const uint64_t nw = (uint64_t)gridDim.x * kWarps;
    for (uint64_t b0 = ((uint64_t)blockIdx.x * kWarps + w) * 32; b0 < a.nb; b0 += nw * 32) {
        uint32_t my_off = 0, my_k = 0;
        if (b0 + lane < a.nb) {
            my_off = a.bloom_off[b0 + lane];
            my_k = a.bloom_off[b0 + lane + 1] - my_off;
        }
        unsigned big = __ballot_sync(kFull, my_k > (uint32_t)kSmall);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1u;
            const uint32_t off = __shfl_sync(kFull, my_off, src), K = __shfl_sync(kFull, my_k, src);
            for (uint32_t i = lane; i < row; i += 32) cur[i] = known[i] = 0;
            __syncwarp();
            uint32_t all_known = 0;  // assigned edges of the bloom
            for (uint32_t i = lane; i < K; i += 32) {
                const uint2 pr = a.pairs[off + i];
                const uint32_t qx = a.place[pr.x & ~kFlag].y, qy = a.place[pr.y & ~kFlag].y;
                const uint32_t qi = qx < qy ? qx : qy, kn = (qx == a.np) + (qy == a.np);
                atomicAdd(&cur[qi], 1u);
                if (kn) atomicAdd(&known[qi], kn);
                all_known += kn;
            }
            all_known = dev::warp_sum(all_known);
            __syncwarp();
            // parts in order, 32 at a time: pairs below; a group for each
            // non-empty part that leaves a butterfly
            uint32_t run = 0, run_known = 0;
            if (lane == 0) gid[a.np] = kNone;
            for (uint32_t i0 = 0; i0 < a.np; i0 += 32) {
                const uint32_t i = i0 + lane;
                const uint32_t n = i < a.np ? cur[i] : 0u;
                const uint32_t incl = dev::warp_incl_scan(n);
                const uint32_t left = K - (run + incl - n);
                run += __shfl_sync(kFull, incl, 31);
                uint32_t higher = 0;  // assigned edges among the pairs of higher parts
                if (a.assigned) {
                    const uint32_t ki = dev::warp_incl_scan(i < a.np ? known[i] : 0u);
                    higher = all_known - run_known - ki;
                    run_known += __shfl_sync(kFull, ki, 31);
                }
                if (i >= a.np) continue;
                const bool g = n > 0u && left >= 2u;
                if constexpr (kPlace) {
                    gid[i] = kNone;
                    if (g) {
                        const uint32_t id = atomicAdd(&a.groups[i], 1u);
                        const uint32_t at = n > 2u ? atomicAdd(&a.members[i], n) : 0u;
                        gid[i] = id;
                        cur[i] = at;
                        size[i] = n;
                        head(a.bl + id, n > 2u ? at : higher, n, left);
                        if (n > 2u) a.bl[id].pair[0].x = higher;
                    }
                } else if (g) {
                    atomicAdd(&t_groups[i], 1u);
                    if (n > 2u) atomicAdd(&t_members[i], n);
                }
            }
            __syncwarp();
            if constexpr (kPlace) {
                for (uint32_t i = lane; i < K; i += 32) {
                    const uint2 pr = a.pairs[off + i];
                    const uint2 x = a.place[pr.x & ~kFlag], y = a.place[pr.y & ~kFlag];
                    const uint32_t qi = x.y < y.y ? x.y : y.y, id = gid[qi];
                    a.sub[off + i] = id;
                    if (id != kNone) {
                        const uint32_t c = atomicAdd(&cur[qi], 1u);
                        if (size[qi] <= 2u) a.bl[id].pair[c] = placed(x, y);
                        else a.out[c] = placed(x, y);
                    }
                }
                __syncwarp();
            }
        }
    }
    if constexpr (!kPlace) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < a.np; i += kT)
            if (t_groups[i]) {
                atomicAdd(&a.groups[i], t_groups[i]);
                atomicAdd(&a.members[i], t_members[i]);
            }
    }
}

// Links per part before the split: room[q] bounds the links part q keeps.
__global__ void __launch_bounds__(kT) k_split_room(const uint64_t *inc_off, const uint2 *place, uint64_t m, uint32_t np,
                                                   unsigned long long *room) {
    __shared__ unsigned long long s_n[kMaxParts];
    for (uint32_t i = threadIdx.x; i < np; i += kT) s_n[i] = 0;
    __syncthreads();
    for (uint64_t e = blockIdx.x * (uint64_t)kT + threadIdx.x; e < m; e += (uint64_t)gridDim.x * kT)
        if (place[e].y < np) atomicAdd(&s_n[place[e].y], (unsigned long long)(inc_off[e + 1] - inc_off[e]));
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < np; i += kT)
        if (s_n[i]) atomicAdd(&room[i], s_n[i]);
}

// One link of an edge in part `part`: whether it is kept (its pair belongs to the
// edge's part and its group holds a butterfly), and as what.
__device__ __forceinline__ bool part_link(uint2 l, uint2 pr, uint32_t s, const uint2 *place, uint32_t part, uint2 &out) {
    const uint2 t = place[(l.y >> 31 ? pr.x : pr.y) & ~kFlag];
    out = make_uint2(t.x | (t.y > part ? kFlag : 0u), s);
    return s != kNone && t.y >= part;
}

// Links of every edge (a warp each): those whose pair belongs to the edge's part,
// as (twin, group), into the part's own range (next: its next free place).  Each
// link costs three scattered reads, which bound this, so a lane has kLU links in
// flight; an edge of more than 32 kLU links is read twice, first to know how many
// it keeps (one link in flight and two readings for all but the smallest: 5.6 ms
// on the 2M-edge graph).
constexpr int kLU = 4;
__global__ void __launch_bounds__(kT) k_split_links(const uint64_t *inc_off, const uint2 *inc, const uint2 *pairs,
                                                    const uint32_t *sub, const uint2 *place, const int *snap,
                                                    uint64_t m, unsigned long long *next, uint2 *out, uint4 *er) {
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const uint64_t nw = ((uint64_t)gridDim.x * kT) >> 5;
    for (uint64_t e = ((uint64_t)blockIdx.x * kT + threadIdx.x) >> 5; e < m; e += nw) {
        const uint64_t lb = inc_off[e], le = inc_off[e + 1];
        const uint2 me = place[e];
        if (me.x == kAssigned) continue;
        const bool once = le - lb <= 32u * kLU;
        uint32_t n = 0;
        unsigned long long at = 0;
        for (int pass = once ? 1 : 0; pass < 2; ++pass) {
            uint32_t k = 0;
            for (uint64_t j0 = lb; j0 < le; j0 += 32u * kLU) {
                uint2 l[kLU], pr[kLU], nl[kLU];
                uint32_t s[kLU], keep[kLU], cnt = 0;
#pragma unroll
                for (int r = 0; r < kLU; ++r) {
                    const uint64_t j = j0 + 32u * r + lane;
                    l[r] = j < le ? inc[j] : make_uint2(0u, 0u);
                }
#pragma unroll
                for (int r = 0; r < kLU; ++r) {
                    const bool in = j0 + 32u * r + lane < le;
                    s[r] = in ? sub[l[r].x] : kNone;
                    pr[r] = in ? pairs[l[r].x] : make_uint2(0u, 0u);
                }
#pragma unroll
                for (int r = 0; r < kLU; ++r) {
                    const bool in = j0 + 32u * r + lane < le;
                    keep[r] = __ballot_sync(kFull, in && part_link(l[r], pr[r], s[r], place, me.y, nl[r]));
                    cnt += __popc(keep[r]);
                }
                if (once) {
                    n = cnt;
                    if (lane == 0 && n) at = atomicAdd(&next[me.y], (unsigned long long)n);
                    at = __shfl_sync(kFull, at, 0);
                }
                if (pass == 1) {
                    uint32_t x = k;
#pragma unroll
                    for (int r = 0; r < kLU; ++r) {
                        if (keep[r] >> lane & 1u) out[at + x + __popc(keep[r] & below)] = nl[r];
                        x += __popc(keep[r]);
                    }
                }
                k += cnt;
            }
            if (pass == 0) {
                n = k;
                if (lane == 0 && n) at = atomicAdd(&next[me.y], (unsigned long long)n);
                at = __shfl_sync(kFull, at, 0);
            }
        }
        if (lane == 0) er[me.x] = make_uint4((uint32_t)at, (uint32_t)(at >> 32), n, (uint32_t)snap[e]);
    }
}

}  // namespace

cudaError_t one_part(const Index &ix, const uint64_t *support, PartGraph &g, int num_sms, Alloc &al) {
    g.m = g.deep = ix.m;
    g.nb = ix.nb;
    g.np = 1;
    g.inc = ix.inc;
    g.pairs = ix.pairs;
    uint32_t *ends = al.get<uint32_t>(4);
    g.part_e = ends;
    g.part_b = ends + 2;
    g.er = al.get<uint4>(ix.m);
    g.bl = al.get<BloomRec>(ix.nb);
    if (al.err != cudaSuccess) return al.err;
    const unsigned wide = (unsigned)num_sms * 16;
    k_edge_rec<<<grid_for(ix.m, 256, wide), 256, 0, al.stream>>>(ix.inc_off, support, ix.m, (uint32_t)ix.nb, ends, g.er);
    al.launches++;
    if (ix.nb) {
        k_bloom_rec<<<grid_for(ix.nb, 256, wide), 256, 0, al.stream>>>(ix.bloom_k, ix.bloom_off, ix.pairs, ix.nb, g.bl);
        al.launches++;
    }
    return cudaGetLastError();
}

static cudaError_t make_parts(const Index &ix, const uint32_t *part, const int *snap, uint32_t np,
                              const uint8_t *assigned, bool skip_first, uint64_t first_rounds, PartGraph &g,
                              int num_sms, Alloc &al) {
    const uint64_t m = ix.m, nb = ix.nb;
    const unsigned wide = (unsigned)num_sms * 16;
    g.deep = m;
    g.assigned = assigned != nullptr;
    g.np = np - skip_first;
    // tables of np + 1 entries, one copy each way: room (64 bits: links of each part,
    // then their first places), first edges, groups and pairs of each part (then
    // their first places, handed out by `cursor`), first blooms, order
    const size_t row = (size_t)np + 1;
    unsigned long long *room = al.get<unsigned long long>(5 * row);
    uint32_t *part_e = reinterpret_cast<uint32_t *>(room + row), *tally = part_e + row;
    uint32_t *cursor = tally, *part_b = tally + 2 * row, *order = part_b + row;
    uint32_t *out_id = al.get<uint32_t>(m);
    g.part_e = part_e;
    g.part_b = part_b;
    g.order = order;
    g.out_id = out_id;
    g.er = al.get<uint4>(m);
    uint32_t *keys = al.get<uint32_t>(m), *tk = al.get<uint32_t>(m), *tv = al.get<uint32_t>(m);
    uint2 *place = al.get<uint2>(m);
    if (al.err != cudaSuccess) return al.err;
    // edges by part
    k_iota2<<<grid_for(m, 256, wide), 256, 0, al.stream>>>(part, assigned, np, m, keys, out_id);
    al.launches++;
    BT_CUDA(radix_sort_u32(keys, out_id, tk, tv, m, bits_for(assigned ? np : np - 1), al));
    k_place<<<grid_for(m, 256, wide), 256, 0, al.stream>>>(keys, out_id, m, np, place, part_e);
    al.launches++;
    al.put(keys);
    al.put(tk);
    al.put(tv);
    // groups and pairs of each part, then their places
    BT_CUDA(cudaMemsetAsync(tally, 0, 8 * row, al.stream));
    BT_CUDA(cudaMemsetAsync(room, 0, 8 * row, al.stream));
    SplitArgs s{ix.bloom_off, nb, ix.pairs, place, np, nullptr, nullptr, nullptr, tally, tally + np + 1,
                assigned != nullptr};
    const size_t smem = sizeof(uint32_t) * (np + 1) * (3 * (kT / 32) + 2);
    // (the attribute belongs to the process: always the same value, so that
    // calls of several threads do not lower one another's)
    const int most = (int)(sizeof(uint32_t) * (kMaxParts + 1) * (3 * (kT / 32) + 2));
    BT_CUDA(cudaFuncSetAttribute(k_split_large<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    BT_CUDA(cudaFuncSetAttribute(k_split_large<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    if (nb) {
        k_split_small<false><<<grid_for(nb, kT, wide), kT, 0, al.stream>>>(s);
        k_split_large<false><<<grid_for(nb, kT, wide), kT, smem, al.stream>>>(s);
        al.launches += 2;
    }
    k_split_room<<<grid_for(m, kT, wide), kT, 0, al.stream>>>(ix.inc_off, place, m, np, room);
    al.launches++;
    BT_CUDA(cudaGetLastError());
    std::vector<unsigned long long> tab(5 * row);
    BT_CUDA(cudaMemcpyAsync(tab.data(), room, 8 * row + 12 * row, cudaMemcpyDeviceToHost, al.stream));
    BT_CUDA(cudaStreamSynchronize(al.stream));
    const std::vector<unsigned long long> hr(tab.begin(), tab.begin() + (long)row);
    uint32_t *he = reinterpret_cast<uint32_t *>(tab.data() + row), *ht = he + row, *hb = ht + 2 * row, *ho = hb + row;
    uint32_t gsum = 0, psum = 0;
    unsigned long long lsum = 0;
    for (uint32_t i = 0; i <= np; ++i) {
        const uint32_t gi = ht[i], pi = ht[row + i];
        hb[i] = ht[i] = gsum;
        ht[row + i] = psum;
        tab[i] = lsum;
        gsum += gi;
        psum += pi;
        lsum += hr[i];
    }
    g.nb = gsum;
    g.m = he[np];
    g.first_e = skip_first ? he[1] : 0u;
    // the heaviest first; those that one block would be long at by a cluster
    const double linked = std::max<double>(1, np - std::count(hr.begin(), hr.begin() + np, 0ull));
    double lim = kHeavy * (double)lsum / linked;
    if (linked < kFewParts) lim = std::min(lim, std::max(kBlockLinks, kHeavy * (double)lsum / kFewParts));
    auto heavy = [&](uint32_t p) { return he[p + 1] - he[p] > kBlockEdges || (double)hr[p] > lim; };
    double longest = 0, its_rounds = 0, rounds = (double)first_rounds;
    for (uint32_t p = skip_first; p < np; ++p) {
        const double links = (double)hr[p], r = rounds_of(links);
        const double t = heavy(p) ? kClusterLinkNs * links + kClusterEdgeNs * (he[p + 1] - he[p]) : kBlockLinkNs * links;
        rounds += r;
        if (t > longest) {
            longest = t;
            its_rounds = r;
        }
    }
    g.lopsided =
        longest > kGridRoundNs * (rounds - its_rounds) + kGridMoreNs * its_rounds + kGridLinkNs * (double)lsum;
    if (g.lopsided) {
        al.put(place);
        return cudaSuccess;
    }
    std::vector<uint32_t> ord(np);
    for (uint32_t i = 0; i < np; ++i) ord[i] = i;
    if (skip_first) ord.erase(ord.begin());
    std::stable_sort(ord.begin(), ord.end(), [&](uint32_t x, uint32_t y) {
        const bool hx = heavy(x), hy = heavy(y);
        return hx != hy ? hx : hr[x] > hr[y];
    });
    for (const uint32_t p : ord) g.n_heavy += heavy(p);
    std::copy(ord.begin(), ord.end(), ho);
    BT_CUDA(cudaMemcpyAsync(room, tab.data(), 40 * row, cudaMemcpyHostToDevice, al.stream));
    uint32_t *sub = al.get<uint32_t>(ix.w2);
    uint2 *pairs = al.get<uint2>(psum), *inc = al.get<uint2>(lsum);
    g.bl = al.get<BloomRec>(gsum);
    g.pairs = pairs;
    g.inc = inc;
    if (al.err != cudaSuccess) return al.err;
    s.out = pairs;
    s.sub = sub;
    s.bl = g.bl;
    s.groups = cursor;
    s.members = cursor + row;
    if (nb) {
        k_split_small<true><<<grid_for(nb, kT, wide), kT, 0, al.stream>>>(s);
        k_split_large<true><<<grid_for(nb, kT, wide), kT, smem, al.stream>>>(s);
        al.launches += 2;
    }
    k_split_links<<<grid_for(m * 32, kT, wide), kT, 0, al.stream>>>(ix.inc_off, ix.inc, ix.pairs, sub, place, snap, m,
                                                                    room, inc, g.er);
    al.launches++;
    BT_CUDA(cudaGetLastError());
    BT_CUDA(cudaStreamSynchronize(al.stream));  // the host tables above
    al.put(place);
    al.put(sub);
    return cudaSuccess;
}

cudaError_t parts_of_ranges(const Index &ix, const uint32_t *part, const int *snap, uint32_t np,
                            const uint8_t *assigned, bool skip_first, uint64_t first_rounds, PartGraph &g,
                            int num_sms, Alloc &al) {
    try {
        return make_parts(ix, part, snap, np, assigned, skip_first, first_rounds, g, num_sms, al);
    } catch (const std::bad_alloc &) {  // the host's tables
        return cudaErrorMemoryAllocation;
    }
}

}  // namespace bt
