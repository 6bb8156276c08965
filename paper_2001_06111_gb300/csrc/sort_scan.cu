// Device-wide exclusive scan and stable LSD radix sort used by the CSR build
// and the BE-Index layout (prefix sums over per-vertex / per-edge counts).
#include "bt_internal.cuh"
#include "bt_device.cuh"

namespace bt {
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanChunk = kScanThreads * kScanItems;

using dev::block_excl_scan;

template <typename T>
__global__ void k_scan_reduce(const T *in, size_t n, T *sums) {
    size_t base = (size_t)blockIdx.x * kScanChunk;
    T acc = 0;
    for (int i = 0; i < kScanItems; ++i) {
        size_t idx = base + (size_t)i * kScanThreads + threadIdx.x;
        if (idx < n) acc += in[idx];
    }
    // block reduce
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    __shared__ T s[kScanThreads / 32];
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        T t = 0;
        for (int i = 0; i < kScanThreads / 32; ++i) t += s[i];
        sums[blockIdx.x] = t;
    }
}

// One block scans the block sums (any count) with a running carry.
template <typename T>
__global__ void k_scan_top(T *sums, size_t nb, T *total) {
    T carry = 0;
    for (size_t base = 0; base < nb; base += kScanThreads) {
        size_t idx = base + threadIdx.x;
        T x = idx < nb ? sums[idx] : T(0);
        T tot;
        T ex = block_excl_scan(x, &tot);
        if (idx < nb) sums[idx] = ex + carry;
        carry += tot;
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

template <typename T>
__global__ void k_scan_down(const T *in, T *out, size_t n, const T *sums) {
    __shared__ T s[kScanChunk];
    size_t base = (size_t)blockIdx.x * kScanChunk;
    for (int i = 0; i < kScanItems; ++i) {
        int li = i * kScanThreads + threadIdx.x;
        size_t idx = base + li;
        s[li] = idx < n ? in[idx] : T(0);
    }
    __syncthreads();
    T v[kScanItems];
    T acc = 0;
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        v[i] = s[threadIdx.x * kScanItems + i];
        acc += v[i];
    }
    T tot;
    T ex = block_excl_scan(acc, &tot) + sums[blockIdx.x];
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) {
        s[threadIdx.x * kScanItems + i] = ex;
        ex += v[i];
    }
    __syncthreads();
    for (int i = 0; i < kScanItems; ++i) {
        int li = i * kScanThreads + threadIdx.x;
        size_t idx = base + li;
        if (idx < n) out[idx] = s[li];
    }
}

template <typename T>
cudaError_t scan_impl(const T *in, T *out, size_t n, T *total, Alloc &al) {
    if (n == 0) {
        if (total) BT_CUDA(cudaMemsetAsync(total, 0, sizeof(T), al.stream));
        return cudaSuccess;
    }
    size_t nb = (n + kScanChunk - 1) / kScanChunk;
    T *sums = al.get<T>(nb);
    if (!sums) return al.err;
    k_scan_reduce<T><<<(unsigned)nb, kScanThreads, 0, al.stream>>>(in, n, sums);
    al.launches++;
    k_scan_top<T><<<1, kScanThreads, 0, al.stream>>>(sums, nb, total);
    al.launches++;
    k_scan_down<T><<<(unsigned)nb, kScanThreads, 0, al.stream>>>(in, out, n, sums);
    al.launches++;
    al.put(sums);
    return cudaGetLastError();
}

// ------------------------------------------------------------- radix sort
constexpr int kSortThreads = 256;
constexpr int kSortRounds = 16;
constexpr int kSortTile = kSortThreads * kSortRounds;

template <typename K>
__global__ void __launch_bounds__(kSortThreads) k_radix_hist(const K *keys, K xin, size_t n, int shift,
                                                             uint32_t *hist, uint32_t ntiles) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const size_t base = (size_t)blockIdx.x * kSortTile;
    K k[kSortRounds];
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r) {
        const size_t idx = base + (size_t)r * kSortThreads + threadIdx.x;
        k[r] = idx < n ? keys[idx] ^ xin : K(0);
    }
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r)
        if (base + (size_t)r * kSortThreads + threadIdx.x < n) atomicAdd(&h[(uint32_t)(k[r] >> shift) & 255u], 1u);
    __syncthreads();
    hist[(size_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter: items of a tile keep their input order within a digit.  A warp
// ranks its 512 neighbouring items by itself (16 turns, counters of its own, no
// block barrier), the tile is put in digit order in shared memory, and every
// digit's run goes out in one piece.  30M 32-bit pairs take 147 us a pass (480 MB
// in and out: 3.3 TB/s), which with the passes that only read or write keys took
// the order of 30M bitruss numbers from 1.51 to 0.86 ms; 60M 64-bit keys take 1.1
// ms a pass, as with four block barriers a turn: their bytes bound it.
template <typename K>
struct SortShared {
    K key[kSortTile];
    uint32_t val[kSortTile];
    uint32_t cnt[kSortThreads / 32][256];  // a warp's counts, then its first place, by digit
    uint32_t start[256], to[256];          // a digit's first place in the tile, and in the output less that
};

// Keys are read xor xin and written xor xout (kout null: not at all); vin null:
// the values are the places.
template <typename K>
__global__ void __launch_bounds__(kSortThreads) k_radix_scatter(const K *kin, K xin, const uint32_t *vin, K *kout,
                                                                K xout, uint32_t *vout, size_t n, int shift,
                                                                const uint32_t *offs, uint32_t ntiles) {
    extern __shared__ __align__(16) unsigned char s_dyn[];
    SortShared<K> &s = *reinterpret_cast<SortShared<K> *>(s_dyn);
    constexpr int kWarps = kSortThreads / 32;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int w = 0; w < kWarps; ++w) s.cnt[w][tid] = 0;
    const uint32_t first = offs[(size_t)tid * ntiles + blockIdx.x];
    __syncthreads();
    const size_t base = (size_t)blockIdx.x * kSortTile, mine = base + (size_t)warp * (32 * kSortRounds) + lane;
    K key[kSortRounds];
    uint32_t val[kSortRounds], rank[kSortRounds];
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r) {
        const size_t idx = mine + 32u * r;
        key[r] = idx < n ? kin[idx] ^ xin : K(0);
        val[r] = idx >= n ? 0u : vin ? vin[idx] : (uint32_t)idx;
    }
    uint32_t *cnt = s.cnt[warp];
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r) {
        const bool valid = mine + 32u * r < n;
        const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
        const uint32_t peers = __match_any_sync(0xffffffffu, valid ? d : 256u);
        const uint32_t before = valid ? cnt[d] : 0u;
        __syncwarp();
        const uint32_t at = __popc(peers & ((1u << lane) - 1u));
        if (valid && at == 0) cnt[d] = before + __popc(peers);
        __syncwarp();
        rank[r] = before + at;
    }
    __syncthreads();
    {
        uint32_t run = 0;
        for (int w = 0; w < kWarps; ++w) {
            const uint32_t c = s.cnt[w][tid];
            s.cnt[w][tid] = run;
            run += c;
        }
        uint32_t total;
        const uint32_t st = block_excl_scan<uint32_t>(run, &total);
        s.start[tid] = st;
        s.to[tid] = first - st;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortRounds; ++r) {
        if (mine + 32u * r >= n) continue;
        const uint32_t d = (uint32_t)(key[r] >> shift) & 255u;
        const uint32_t pos = s.start[d] + cnt[d] + rank[r];
        s.key[pos] = key[r];
        s.val[pos] = val[r];
    }
    __syncthreads();
    const uint32_t have = n - base < (size_t)kSortTile ? (uint32_t)(n - base) : (uint32_t)kSortTile;
    for (uint32_t i = tid; i < have; i += kSortThreads) {
        const K k = s.key[i];
        const uint32_t pos = s.to[(uint32_t)(k >> shift) & 255u] + i;
        if (kout) kout[pos] = k ^ xout;
        vout[pos] = s.val[i];
    }
}

template <typename K>
cudaError_t radix_impl(K *keys, uint32_t *vals, K *tk, uint32_t *tv, size_t n, int bits,
                       Alloc &al) {
    if (n <= 1 || bits <= 0) return cudaSuccess;
    uint32_t ntiles = (uint32_t)((n + kSortTile - 1) / kSortTile);
    uint32_t *hist = al.get<uint32_t>((size_t)256 * ntiles);
    if (!hist) return al.err;
    K *ka = keys, *kb = tk;
    uint32_t *va = vals, *vb = tv;
    int passes = (bits + 7) / 8;
    BT_CUDA(cudaFuncSetAttribute(k_radix_scatter<K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(SortShared<K>)));
    for (int p = 0; p < passes; ++p) {
        int shift = 8 * p;
        k_radix_hist<K><<<ntiles, kSortThreads, 0, al.stream>>>(ka, K(0), n, shift, hist, ntiles);
        al.launches++;
        cudaError_t e = scan_impl<uint32_t>(hist, hist, (size_t)256 * ntiles, nullptr, al);
        if (e != cudaSuccess) return e;
        k_radix_scatter<K><<<ntiles, kSortThreads, sizeof(SortShared<K>), al.stream>>>(ka, K(0), va, kb, K(0), vb, n,
                                                                                       shift, hist, ntiles);
        al.launches++;
        K *t = ka; ka = kb; kb = t;
        uint32_t *u = va; va = vb; vb = u;
    }
    if (ka != keys) {
        BT_CUDA(cudaMemcpyAsync(keys, ka, n * sizeof(K), cudaMemcpyDeviceToDevice, al.stream));
        BT_CUDA(cudaMemcpyAsync(vals, va, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, al.stream));
    }
    al.put(hist);
    return cudaGetLastError();
}

__global__ void k_widen(const uint32_t *in, uint64_t *out, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        out[i] = in[i];
}

}  // namespace

cudaError_t widen_u32(const uint32_t *in, uint64_t *out, size_t n, Alloc &al) {
    if (n == 0) return cudaSuccess;
    size_t g = (n + 255) / 256;
    if (g > 152 * 64) g = 152 * 64;
    k_widen<<<(unsigned)g, 256, 0, al.stream>>>(in, out, n);
    al.launches++;
    return cudaGetLastError();
}

cudaError_t exclusive_scan_u32(const uint32_t *in, uint32_t *out, size_t n, uint32_t *total,
                               Alloc &al) {
    return scan_impl<uint32_t>(in, out, n, total, al);
}
cudaError_t exclusive_scan_u64(const uint64_t *in, uint64_t *out, size_t n, uint64_t *total,
                               Alloc &al) {
    return scan_impl<uint64_t>(in, out, n, total, al);
}
cudaError_t radix_sort_u32(uint32_t *keys, uint32_t *vals, uint32_t *tk, uint32_t *tv, size_t n,
                           int bits, Alloc &al) {
    return radix_impl<uint32_t>(keys, vals, tk, tv, n, bits, al);
}
cudaError_t radix_order_desc_u32(const uint32_t *keys, size_t n, uint32_t *order, uint32_t *sorted, Alloc &al) {
    if (n == 0) return cudaSuccess;
    if (n == 1) {  // in order as it is (the passes: 0.13 against 0.04 ms)
        if (sorted) BT_CUDA(cudaMemcpyAsync(sorted, keys, sizeof(uint32_t), cudaMemcpyDeviceToDevice, al.stream));
        return cudaMemsetAsync(order, 0, sizeof(uint32_t), al.stream);
    }
    const uint32_t ntiles = (uint32_t)((n + kSortTile - 1) / kSortTile);
    uint32_t *hist = al.get<uint32_t>((size_t)256 * ntiles);
    uint32_t *ka = al.get<uint32_t>(n), *va = al.get<uint32_t>(n), *kb = al.get<uint32_t>(n);
    if (al.err != cudaSuccess) return al.err;
    const size_t smem = sizeof(SortShared<uint32_t>);
    BT_CUDA(cudaFuncSetAttribute(k_radix_scatter<uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // keys -> a -> (kb, order) -> a -> (sorted, order)
    for (int p = 0; p < 4; ++p) {
        const uint32_t *kin = p == 0 ? keys : p == 2 ? kb : ka, *vin = p == 0 ? nullptr : p == 2 ? order : va;
        uint32_t *kout = p == 3 ? sorted : p == 1 ? kb : ka, *vout = p & 1 ? order : va;
        const uint32_t xin = p == 0 ? ~0u : 0u, xout = p == 3 ? ~0u : 0u;
        k_radix_hist<uint32_t><<<ntiles, kSortThreads, 0, al.stream>>>(kin, xin, n, 8 * p, hist, ntiles);
        cudaError_t e = scan_impl<uint32_t>(hist, hist, (size_t)256 * ntiles, nullptr, al);
        if (e != cudaSuccess) return e;
        k_radix_scatter<uint32_t><<<ntiles, kSortThreads, smem, al.stream>>>(kin, xin, vin, kout, xout, vout, n, 8 * p,
                                                                             hist, ntiles);
        al.launches += 2;
    }
    al.put(hist);
    al.put(ka);
    al.put(va);
    al.put(kb);
    return cudaGetLastError();
}
cudaError_t radix_sort_u64(uint64_t *keys, uint32_t *vals, uint64_t *tk, uint32_t *tv, size_t n,
                           int bits, Alloc &al) {
    return radix_impl<uint64_t>(keys, vals, tk, tv, n, bits, al);
}

}  // namespace bt
