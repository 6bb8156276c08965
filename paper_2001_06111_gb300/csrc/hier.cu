// Bitruss hierarchy from the bitruss numbers (Defs. 4-5, Section II).
//
// The k-bitrusses are nested (H_{k+1} satisfies the support bound of H_k, and
// H_k is the unique maximal subgraph that does), and an edge lies in H_k
// exactly when phi_e >= k.  So one stable sort of the edges by phi, largest
// first, lists every H_k as a prefix, and H_k alone is a stream compaction of
// the edges with phi_e >= k.
#include "bt_device.cuh"
#include "bt_internal.cuh"

namespace bt {
namespace {

constexpr int kHT = 256, kHR = 16, kHTile = kHT * kHR;

// Entries >= k of each tile of kHTile.
__global__ void __launch_bounds__(kHT) k_count_ge(const uint32_t *phi, uint64_t m, uint32_t k, uint32_t *count) {
    const uint64_t base = (uint64_t)blockIdx.x * kHTile;
    uint32_t n = 0;
#pragma unroll
    for (int r = 0; r < kHR; ++r) {
        const uint64_t i = base + (uint64_t)r * kHT + threadIdx.x;
        n += i < m && phi[i] >= k;
    }
    n = dev::block_sum(n);
    if (threadIdx.x == 0) count[blockIdx.x] = n;
}

// Their places, ascending: a warp takes 512 neighbouring entries.
__global__ void __launch_bounds__(kHT) k_write_ge(const uint32_t *phi, uint64_t m, uint32_t k, const uint32_t *first,
                                                  uint32_t *out) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t base = (uint64_t)blockIdx.x * kHTile + warp * (32 * kHR);
    unsigned mask[kHR];
    uint32_t n = 0;
#pragma unroll
    for (int r = 0; r < kHR; ++r) {
        const uint64_t i = base + 32u * r + lane;
        mask[r] = __ballot_sync(0xffffffffu, i < m && phi[i] >= k);
        n += __popc(mask[r]);
    }
    __shared__ uint32_t s_n[kHT / 32];
    if (lane == 0) s_n[warp] = n;
    __syncthreads();
    uint32_t at = first[blockIdx.x];
    for (uint32_t w = 0; w < warp; ++w) at += s_n[w];
#pragma unroll
    for (int r = 0; r < kHR; ++r) {
        if (mask[r] >> lane & 1u) out[at + __popc(mask[r] & ((1u << lane) - 1u))] = (uint32_t)(base + 32u * r + lane);
        at += __popc(mask[r]);
    }
}

}  // namespace

cudaError_t hierarchy_order(const uint32_t *phi, uint64_t m, uint32_t *order, uint32_t *phi_sorted, Alloc &al) {
    return radix_order_desc_u32(phi, m, order, phi_sorted, al);
}

cudaError_t select_ge(const uint32_t *phi, uint64_t m, uint32_t k, uint32_t *out, uint32_t *d_count,
                      Alloc &al) {
    if (m == 0) return cudaMemsetAsync(d_count, 0, sizeof(uint32_t), al.stream);
    const uint32_t tiles = (uint32_t)((m + kHTile - 1) / kHTile);
    uint32_t *count = al.get<uint32_t>(tiles);
    if (al.err != cudaSuccess) return al.err;
    k_count_ge<<<tiles, kHT, 0, al.stream>>>(phi, m, k, count);
    al.launches++;
    BT_CUDA(exclusive_scan_u32(count, count, tiles, d_count, al));
    k_write_ge<<<tiles, kHT, 0, al.stream>>>(phi, m, k, count, out);
    al.launches++;
    al.put(count);
    return cudaGetLastError();
}

}  // namespace bt
