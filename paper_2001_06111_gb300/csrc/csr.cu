// Degree, priority rank and rank-ordered CSR (the preprocessing of Alg. 3:
// "compute p(u) for each u", Def. 7), plus the per-arc wedge prefix lengths
// that bound the priority-obeyed wedge loops (Def. 10, Lemma 6).
#include "bt_device.cuh"
#include "bt_internal.cuh"

namespace bt {
namespace {

// Global id of each endpoint.  Section II assumes every upper id exceeds
// every lower id: lower v -> v, upper u -> nL + u.  BT_TIE_LOWER_FIRST swaps
// the layers (upper u -> u, lower v -> nU + v).
__device__ __forceinline__ void gids(int32_t u, int32_t v, uint32_t nU, uint32_t nL, uint32_t flags,
                                     uint32_t &gu, uint32_t &gv) {
    if (flags & BT_TIE_LOWER_FIRST) {
        gu = (uint32_t)u;
        gv = nU + (uint32_t)v;
    } else {
        gu = nL + (uint32_t)u;
        gv = (uint32_t)v;
    }
}

__global__ void k_degree(const int32_t *edges, uint64_t m, uint32_t nU, uint32_t nL, uint32_t flags,
                         uint32_t *deg, uint32_t *err) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m;
         i += (uint64_t)gridDim.x * blockDim.x) {
        int2 e = reinterpret_cast<const int2 *>(edges)[i];
        if (e.x < 0 || e.y < 0 || (uint32_t)e.x >= nU || (uint32_t)e.y >= nL) {
            atomicOr(err, kErrRange);
            continue;
        }
        uint32_t gu, gv;
        gids(e.x, e.y, nU, nL, flags, gu, gv);
        atomicAdd(&deg[gu], 1u);
        atomicAdd(&deg[gv], 1u);
    }
}

__global__ void k_iota(uint32_t *a, uint32_t n) {
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        a[i] = i;
}

// order[r] = global id of rank r (sorted by degree, stable on id => ties by
// id); deg_sorted[r] = its degree.
__global__ void k_rank(const uint32_t *order, const uint32_t *deg_sorted, uint32_t n,
                       uint32_t *rank, uint64_t *degr) {
    for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
        rank[order[r]] = r;
        degr[r] = deg_sorted[r];
    }
}

// Union ranking key of every vertex id: its graph, then its degree (the sort
// is stable, so ties stay in id order, as for the graph alone).
__global__ void k_graph_keys(const uint32_t *deg, uint32_t n, uint32_t nU, uint32_t nL, uint32_t flags,
                             uint32_t ng, const uint32_t *offU, const uint32_t *offL, int dbits,
                             uint32_t *keys) {
    for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < n; x += gridDim.x * blockDim.x) {
        // the layer and layer-local id of x (see gids)
        bool upper;
        uint32_t loc;
        if (flags & BT_TIE_LOWER_FIRST) {
            upper = x < nU;
            loc = upper ? x : x - nU;
        } else {
            upper = x >= nL;
            loc = upper ? x - nL : x;
        }
        const uint32_t *off = upper ? offU : offL;
        uint32_t lo = 0, hi = ng;  // largest g with off[g] <= loc
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (off[mid] <= loc) lo = mid; else hi = mid;
        }
        keys[x] = lo << dbits | deg[x];
    }
}

// After the union sort: rank r's degree and the first rank of its graph.
__global__ void k_graph_rank(const uint32_t *keys_sorted, uint32_t n, int dbits, const uint32_t *offU,
                             const uint32_t *offL, uint32_t *deg_sorted, uint32_t *vbase) {
    for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
        const uint32_t k = keys_sorted[r];
        const uint32_t gi = k >> dbits;
        deg_sorted[r] = k & ((1u << dbits) - 1u);
        vbase[r] = offU[gi] + offL[gi];  // vertices of the graphs before it
    }
}

__global__ void k_arcs(const int32_t *edges, uint64_t m, uint32_t nU, uint32_t nL, uint32_t flags,
                       const uint32_t *rank, uint32_t n, uint64_t *keys, uint32_t *vals) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m;
         i += (uint64_t)gridDim.x * blockDim.x) {
        int2 e = reinterpret_cast<const int2 *>(edges)[i];
        if (e.x < 0 || e.y < 0 || (uint32_t)e.x >= nU || (uint32_t)e.y >= nL) {
            keys[2 * i] = keys[2 * i + 1] = 0;  // flagged by k_degree; call fails
            vals[2 * i] = vals[2 * i + 1] = (uint32_t)i;
            continue;
        }
        uint32_t gu, gv;
        gids(e.x, e.y, nU, nL, flags, gu, gv);
        uint64_t ru = rank[gu], rv = rank[gv];
        keys[2 * i] = ru * n + rv;
        vals[2 * i] = (uint32_t)i;
        keys[2 * i + 1] = rv * n + ru;
        vals[2 * i + 1] = (uint32_t)i;
    }
}

// Arc j of the sorted keys: its row, its end, its edge.  low[e]: place of edge e in
// the list of its lower-ranked endpoint v, i.e. how many neighbours of v rank
// below the other endpoint.  hv[u]: the length of u's prefix of lower-ranked
// neighbours (zeroed before).
__global__ void k_csr_fill(const uint64_t *keys, const uint32_t *vals, uint64_t na, uint32_t n, const uint64_t *off,
                           uint32_t *row_of, uint32_t *adj, uint32_t *eid, uint32_t *low, uint32_t *hv, uint32_t *err) {
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < na;
         j += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t k = keys[j];
        const uint32_t row = (uint32_t)(k / n), col = (uint32_t)(k - (uint64_t)row * n), e = vals[j];
        row_of[j] = row;
        adj[j] = col;
        eid[j] = e;
        if (col > row) {
            low[e] = (uint32_t)(j - off[row]);
        } else {
            // the last of the prefix: the next arc leaves it
            const uint64_t nx = j + 1 < na ? keys[j + 1] : ~0ull;
            if (nx > (uint64_t)row * n + row) hv[row] = (uint32_t)(j + 1 - off[row]);
        }
        if (j > 0 && keys[j - 1] == k) atomicOr(err, kErrDup);
    }
}

// A thread per arc (u, v), v < u: pl = |{w in N(v): w < u}|, the place of u in N(v);
// its edge gets the internal id hoff[u] + its place in u's prefix; wv[u] (zeroed
// before) += pl, one atomic for the arcs of u in a warp.  (A warp per vertex left
// one warp with the largest vertex's list: 12 + 6 ms on the 30M-edge graph.)
__global__ void k_wedge_prefix(const uint64_t *off, const uint32_t *row_of, const uint32_t *adj, uint32_t *eid,
                               const uint32_t *low, const uint32_t *hoff, uint64_t na, uint32_t *pl,
                               unsigned long long *wv, uint32_t *newid) {
    const int lane = threadIdx.x & 31;
    for (uint64_t j0 = blockIdx.x * (uint64_t)blockDim.x; j0 < na; j0 += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t j = j0 + threadIdx.x;
        uint32_t u = 0xFFFFFFFFu;
        unsigned long long p = 0;
        if (j < na) {
            u = row_of[j];
            if (adj[j] < u) {
                const uint32_t e = eid[j], id = hoff[u] + (uint32_t)(j - off[u]);
                p = low[e];
                pl[j] = (uint32_t)p;
                newid[e] = id;
                eid[j] = id;
            }
        }
        // arcs of a vertex are neighbours: sums by a segmented scan
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, p, o);
            const uint32_t v = __shfl_up_sync(0xffffffffu, u, o);
            if (lane >= o && v == u) p += y;
        }
        const uint32_t nu = __shfl_down_sync(0xffffffffu, u, 1);
        if (p && (lane == 31 || nu != u)) atomicAdd(&wv[u], p);
    }
}

// Internal ids of the other arcs, and the places of the neighbours (Csr::wplace) if asked for.
__global__ void k_relabel(const uint32_t *row_of, const uint32_t *adj, uint64_t na, uint32_t *eid, const uint32_t *newid,
                          const uint32_t *place, uint32_t *wplace) {
    for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < na;
         j += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t v = adj[j];
        if (v > row_of[j]) eid[j] = newid[eid[j]];
        if (place) wplace[j] = place[v];
    }
}

// Layer of the vertex of each rank: 1 for the ids from `first` on.
__global__ void k_layer(const uint32_t *order, uint32_t n, uint32_t first, uint32_t *layer) {
    for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x)
        layer[r] = order[r] >= first;
}
// ones[r]: vertices of layer 1 below rank r.
__global__ void k_place_in_layer(const uint32_t *layer, const uint32_t *ones, uint32_t n, uint32_t *place) {
    for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x)
        place[r] = layer[r] ? ones[r] : r - ones[r];
}

// Start vertices that get a block each, by the power of two of their wedges: the
// counting kernels take the heaviest first, so that none is begun when the other
// blocks are done.  tab[0 .. 64): how many of each class, [64]: of all, [65 .. 129):
// placed.  all: the sum of the wedges (a scan and a copy of its own before).
__device__ __forceinline__ uint32_t wedge_class(uint64_t W) { return (uint32_t)__clzll((long long)W); }
__global__ void k_heavy_count(const uint64_t *wv, const uint32_t *hv, uint32_t n, uint32_t *tab, uint64_t *all) {
    __shared__ uint32_t s_n[64];
    if (threadIdx.x < 64) s_n[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long sum = 0;
    for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
        const uint64_t W = wv[u];
        sum += W;
        if (W && !is_light(W, hv[u])) atomicAdd(&s_n[wedge_class(W)], 1u);
    }
    sum = dev::block_sum(sum);
    if (threadIdx.x == 0 && sum) atomicAdd(reinterpret_cast<unsigned long long *>(all), sum);
    if (threadIdx.x < 64 && s_n[threadIdx.x]) {
        atomicAdd(&tab[threadIdx.x], s_n[threadIdx.x]);
        atomicAdd(&tab[64], s_n[threadIdx.x]);
    }
}
__global__ void k_heavy_place(const uint64_t *wv, const uint32_t *hv, uint32_t n, uint32_t *tab, uint32_t *heavy) {
    __shared__ uint32_t s_first[64];
    if (threadIdx.x == 0) {
        uint32_t run = 0;
        for (int c = 0; c < 64; ++c) {
            s_first[c] = run;
            run += tab[c];
        }
    }
    __syncthreads();
    for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < n; u += gridDim.x * blockDim.x) {
        const uint64_t W = wv[u];
        if (W && !is_light(W, hv[u])) {
            const uint32_t c = wedge_class(W);
            heavy[s_first[c] + atomicAdd(&tab[65 + c], 1u)] = u;
        }
    }
}

template <typename T>
__global__ void k_gather(const T *in, const uint32_t *newid, T *out, uint64_t m) {
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < m;
         e += (uint64_t)gridDim.x * blockDim.x)
        out[e] = in[newid[e]];
}

__global__ void k_scatter_u8(const uint8_t *in, const uint32_t *newid, uint8_t *out, uint64_t m) {
    for (uint64_t e = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; e < m;
         e += (uint64_t)gridDim.x * blockDim.x)
        out[newid[e]] = in[e];
}

inline unsigned grid_for(uint64_t items, int threads, unsigned cap = 152 * 32) {
    uint64_t g = (items + threads - 1) / threads;
    if (g == 0) g = 1;
    return (unsigned)(g < cap ? g : cap);
}

// Relabels a concatenation of independent graphs into one disjoint union:
// edge i of graph g gets its upper id shifted by offU[g] and its lower id by
// offL[g].  Ids are checked against the graph's own layer sizes first; the
// lowest failing graph index is kept in *bad_graph.
__global__ void k_union(int32_t *edges, uint64_t m_total, const uint64_t *goff, uint32_t ng,
                        const uint32_t *offU, const uint32_t *offL, const uint32_t *gnU,
                        const uint32_t *gnL, uint32_t *err, uint32_t *bad_graph) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m_total;
         i += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t lo = 0, hi = ng;  // largest g with goff[g] <= i
        while (hi - lo > 1) {
            uint32_t mid = (lo + hi) >> 1;
            if (goff[mid] <= i) lo = mid; else hi = mid;
        }
        const uint32_t g = lo;
        int2 e = reinterpret_cast<int2 *>(edges)[i];
        if (e.x < 0 || e.y < 0 || (uint32_t)e.x >= gnU[g] || (uint32_t)e.y >= gnL[g]) {
            atomicOr(err, kErrRange);
            atomicMin(bad_graph, g);
            continue;
        }
        e.x += (int32_t)offU[g];
        e.y += (int32_t)offL[g];
        reinterpret_cast<int2 *>(edges)[i] = e;
    }
}

}  // namespace

cudaError_t union_edges(int32_t *d_edges, uint64_t m_total, const uint64_t *d_goff, uint32_t ng,
                        const uint32_t *d_offU, const uint32_t *d_offL, const uint32_t *d_nU,
                        const uint32_t *d_nL, uint32_t *err_word, uint32_t *bad_graph, Alloc &al) {
    if (m_total == 0) return cudaSuccess;
    k_union<<<grid_for(m_total, 256), 256, 0, al.stream>>>(d_edges, m_total, d_goff, ng, d_offU,
                                                           d_offL, d_nU, d_nL, err_word, bad_graph);
    al.launches++;
    return cudaGetLastError();
}

cudaError_t build_csr(const int32_t *d_edges, uint64_t m, uint32_t nU, uint32_t nL, uint32_t flags,
                      Csr &g, uint32_t *err_word, Alloc &al, const GraphSplit *split) {
    const uint32_t n = nU + nL;
    g.n = n;
    g.m = m;
    g.cnt_n = n;
    // graph-by-graph ranking when graph and degree fit one 32-bit key
    const int dbits = split ? bits_for(split->max_n) : 0;
    const int gbits = split ? bits_for(split->ng > 0 ? split->ng - 1 : 0) : 0;
    const bool by_graph = split && split->ng > 1 && dbits + gbits <= 32 && dbits < 32;
    uint32_t *deg = al.get<uint32_t>(n);
    uint32_t *order = al.get<uint32_t>(n);
    uint32_t *tk = al.get<uint32_t>(n);
    uint32_t *tv = al.get<uint32_t>(n);
    uint32_t *rank = al.get<uint32_t>(n);
    uint64_t *degr = al.get<uint64_t>((size_t)n + 1);
    g.off = al.get<uint64_t>((size_t)n + 1);
    if (al.err != cudaSuccess) return al.err;
    al.mark(kPhCsr, false);
    BT_CUDA(cudaMemsetAsync(deg, 0, sizeof(uint32_t) * n, al.stream));
    k_degree<<<grid_for(m, 256), 256, 0, al.stream>>>(d_edges, m, nU, nL, flags, deg, err_word);
    al.launches++;
    k_iota<<<grid_for(n, 256), 256, 0, al.stream>>>(order, n);
    al.launches++;
    if (by_graph) {
        uint32_t *gkey = al.get<uint32_t>(n);
        g.vbase = al.get<uint32_t>(n);
        if (al.err != cudaSuccess) return al.err;
        k_graph_keys<<<grid_for(n, 256), 256, 0, al.stream>>>(deg, n, nU, nL, flags, split->ng, split->offU,
                                                              split->offL, dbits, gkey);
        al.launches++;
        BT_CUDA(radix_sort_u32(gkey, order, tk, tv, n, dbits + gbits, al));
        k_graph_rank<<<grid_for(n, 256), 256, 0, al.stream>>>(gkey, n, dbits, split->offU, split->offL, deg,
                                                              g.vbase);
        al.launches++;
        al.put(gkey);
        g.cnt_n = split->max_n;
    } else {
        // degrees are <= max(nU, nL); a stable sort on degree keeps ties in id order
        BT_CUDA(radix_sort_u32(deg, order, tk, tv, n, bits_for(nU > nL ? nU : nL), al));
    }
    // deg now holds the degrees in rank order
    BT_CUDA(cudaMemsetAsync(degr, 0, sizeof(uint64_t) * ((size_t)n + 1), al.stream));
    k_rank<<<grid_for(n, 256), 256, 0, al.stream>>>(order, deg, n, rank, degr);
    al.launches++;
    BT_CUDA(cudaGetLastError());
    al.put(tk);
    al.put(tv);
    // off = exclusive scan of degree by rank
    BT_CUDA(exclusive_scan_u64(degr, g.off, (size_t)n + 1, nullptr, al));

    const uint64_t na = 2 * m;
    uint64_t *keys = al.get<uint64_t>(na);
    uint32_t *vals = al.get<uint32_t>(na);
    uint64_t *k2 = al.get<uint64_t>(na);
    uint32_t *v2 = al.get<uint32_t>(na);
    if (al.err != cudaSuccess) return al.err;
    k_arcs<<<grid_for(m, 256), 256, 0, al.stream>>>(d_edges, m, nU, nL, flags, rank, n, keys, vals);
    al.launches++;
    BT_CUDA(radix_sort_u64(keys, vals, k2, v2, na, bits_for((uint64_t)n * n - 1), al));
    al.put(k2);
    al.put(v2);
    g.adj = al.get<uint32_t>(na);
    g.eid = al.get<uint32_t>(na);
    g.pl = al.get<uint32_t>(na);
    g.hv = al.get<uint32_t>(n);
    g.wv = al.get<uint64_t>(n);
    g.heavy = al.get<uint32_t>(n);
    g.n_heavy = al.get<uint32_t>(129);
    g.totals = al.get<uint64_t>(5);
    g.newid = al.get<uint32_t>(m);
    uint32_t *low = al.get<uint32_t>(m), *hoff = al.get<uint32_t>(n), *row_of = al.get<uint32_t>(na);
    if (al.err != cudaSuccess) return al.err;
    BT_CUDA(cudaMemsetAsync(g.hv, 0, sizeof(uint32_t) * n, al.stream));
    BT_CUDA(cudaMemsetAsync(g.wv, 0, sizeof(uint64_t) * n, al.stream));
    BT_CUDA(cudaMemsetAsync(g.totals, 0, sizeof(uint64_t) * 5, al.stream));
    BT_CUDA(cudaMemsetAsync(g.n_heavy, 0, sizeof(uint32_t) * 129, al.stream));
    k_csr_fill<<<grid_for(na, 256), 256, 0, al.stream>>>(keys, vals, na, n, g.off, row_of, g.adj, g.eid, low, g.hv,
                                                         err_word);
    al.launches++;
    al.put(keys);
    al.put(vals);
    // internal edge ids grouped by the higher-ranked endpoint
    BT_CUDA(exclusive_scan_u32(g.hv, hoff, n, nullptr, al));
    k_wedge_prefix<<<grid_for(na, 256), 256, 0, al.stream>>>(g.off, row_of, g.adj, g.eid, low, hoff, na, g.pl,
                                                             reinterpret_cast<unsigned long long *>(g.wv), g.newid);
    // (a fixed arena has no room for it)
    if (!g.vbase && n > kPlacesFrom && !al.arena) {
        g.place = al.get<uint32_t>(n);
        g.wplace = al.get<uint32_t>(na);
        uint32_t *layer = al.get<uint32_t>(n), *ones = al.get<uint32_t>(n);
        if (al.err != cudaSuccess) return al.err;
        const bool upper_first = (flags & BT_TIE_LOWER_FIRST) != 0;
        k_layer<<<grid_for(n, 256), 256, 0, al.stream>>>(order, n, upper_first ? nU : nL, layer);
        BT_CUDA(exclusive_scan_u32(layer, ones, n, nullptr, al));
        k_place_in_layer<<<grid_for(n, 256), 256, 0, al.stream>>>(layer, ones, n, g.place);
        al.launches += 2;
        al.put(layer);
        al.put(ones);
        g.cnt_n = nU > nL ? nU : nL;
    }
    k_relabel<<<grid_for(na, 256), 256, 0, al.stream>>>(row_of, g.adj, na, g.eid, g.newid, g.place, g.wplace);
    k_heavy_count<<<grid_for(n, 256, 152 * 4), 256, 0, al.stream>>>(g.wv, g.hv, n, g.n_heavy, g.totals);
    k_heavy_place<<<grid_for(n, 256, 152 * 4), 256, 0, al.stream>>>(g.wv, g.hv, n, g.n_heavy, g.heavy);
    al.launches += 4;
    al.put(low);
    al.put(hoff);
    al.put(row_of);
    al.mark(kPhCsr, true);
    al.put(deg);
    al.put(order);
    al.put(rank);
    al.put(degr);
    return cudaGetLastError();
}

cudaError_t gather_u64(const uint64_t *in, const uint32_t *newid, uint64_t *out, uint64_t m, Alloc &al) {
    if (m == 0) return cudaSuccess;
    k_gather<uint64_t><<<grid_for(m, 256), 256, 0, al.stream>>>(in, newid, out, m);
    al.launches++;
    return cudaGetLastError();
}

cudaError_t gather_u32(const uint32_t *in, const uint32_t *newid, uint32_t *out, uint64_t m, Alloc &al) {
    if (m == 0) return cudaSuccess;
    k_gather<uint32_t><<<grid_for(m, 256), 256, 0, al.stream>>>(in, newid, out, m);
    al.launches++;
    return cudaGetLastError();
}

cudaError_t scatter_u8(const uint8_t *in, const uint32_t *newid, uint8_t *out, uint64_t m, Alloc &al) {
    if (m == 0) return cudaSuccess;
    k_scatter_u8<<<grid_for(m, 256), 256, 0, al.stream>>>(in, newid, out, m);
    al.launches++;
    return cudaGetLastError();
}

// Frees the CSR (and newid unless a caller took it over).
void free_csr(Csr &g, Alloc &al) {
    al.put(g.newid);
    al.put(g.vbase);
    al.put(g.place);
    al.put(g.wplace);
    al.put(g.off);
    al.put(g.adj);
    al.put(g.eid);
    al.put(g.pl);
    al.put(g.hv);
    al.put(g.wv);
    al.put(g.heavy);
    al.put(g.n_heavy);
    al.put(g.totals);
    g = Csr{};
}

}  // namespace bt
