// Block- and warp-level helpers shared by the kernels of libbitruss.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace bt {
namespace dev {

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Exclusive scan of one value per thread over a block of <= 1024 threads;
// the block total is returned through *total.  Contains __syncthreads().
template <typename T>
__device__ T block_excl_scan(T x, T *total) {
    __shared__ T s_warp[32];
    __shared__ T s_total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    T inc = warp_incl_scan(x);
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T v = lane < nwarps ? s_warp[lane] : T(0);
        T vi = warp_incl_scan(v);
        if (lane < nwarps) s_warp[lane] = vi - v;
        if (lane == nwarps - 1) s_total = vi;
    }
    __syncthreads();
    T res = inc - x + s_warp[warp];
    *total = s_total;
    __syncthreads();
    return res;
}

// Sum over the block (result valid in every thread).  Contains __syncthreads().
template <typename T>
__device__ T block_sum(T x) {
    __shared__ T s_part[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    x = warp_sum(x);
    if (lane == 0) s_part[warp] = x;
    __syncthreads();
    T t = 0;
    for (int i = 0; i < nwarps; ++i) t += s_part[i];
    __syncthreads();
    return t;
}

__device__ __forceinline__ uint32_t lower_bound_u32(const uint32_t *a, uint32_t len, uint32_t key) {
    uint32_t lo = 0, hi = len;
    while (lo < hi) {
        uint32_t mid = (lo + hi) >> 1;
        if (a[mid] < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Largest index i in [0, len) with a[i] <= key (a sorted ascending, a[0] <= key).
__device__ __forceinline__ uint32_t last_le_u32(const uint32_t *a, uint32_t len, uint32_t key) {
    uint32_t lo = 0, hi = len;  // answer in [lo, hi)
    while (hi - lo > 1) {
        uint32_t mid = (lo + hi) >> 1;
        if (a[mid] <= key) lo = mid; else hi = mid;
    }
    return lo;
}

// Items of different lengths laid side by side: off[0 .. n] (shared memory) are
// their first entries, strictly ascending, off[n] the number of entries.  A warp
// takes neighbouring entries, 32 at a turn, and finds the items of all of them
// from 32 neighbouring offsets read once; a binary search an entry (ten
// conflicting reads of shared memory) was what bound such loops.

// The item that holds entry x (the same for the whole warp).
__device__ __forceinline__ uint32_t item_of(const uint32_t *off, uint32_t n, uint32_t x) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t b = 0;  // n <= 1024: first the 32 items it lies among
    if (n > 32u)
        b = 32u * (uint32_t)(__popc(__ballot_sync(0xffffffffu, 32u * lane < n && off[32u * lane] <= x)) - 1);
    return b + (uint32_t)__popc(__ballot_sync(0xffffffffu, b + lane < n && off[b + lane] <= x)) - 1u;
}
// The items of entries [w, w + 32), one a lane; j0: the item of entry w, which
// becomes that of w + 32.
__device__ __forceinline__ uint32_t items_of(const uint32_t *off, uint32_t n, uint32_t w, uint32_t &j0) {
    const uint32_t lane = threadIdx.x & 31, i = j0 + 1u + lane;
    const uint32_t rel = i <= n ? off[i] - w : 64u;
    const unsigned starts = __reduce_or_sync(0xffffffffu, rel < 32u ? 1u << rel : 0u);
    const uint32_t j = j0 + __popc(starts & (0xffffffffu >> (31u - lane)));
    j0 += __popc(__ballot_sync(0xffffffffu, rel <= 32u));
    return j;
}
// Entries [lo, hi) of `total` that warp `w` of `nw` takes.
__device__ __forceinline__ void share_of(uint32_t total, uint32_t w, uint32_t nw, uint32_t &lo, uint32_t &hi) {
    const uint32_t per = ((total + nw * 32u - 1u) / (nw * 32u)) * 32u;
    lo = w * per < total ? w * per : total;
    hi = total - lo < per ? total : lo + per;
}

}  // namespace dev
}  // namespace bt
