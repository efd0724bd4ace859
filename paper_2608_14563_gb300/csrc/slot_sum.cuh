// slot_sum.cuh -- fp64 totals of the per-warp partial sums that a GEMM's epilogue leaves
// (groups of N floats, one per slot), by a cluster of blocks per layer.
//
// GB300 adds two fp64 numbers per SM and clock at best: one block adding the 17,280 pairs
// of a 3072 x 23040 layer took 27 us, a cluster of kSlotBlocks spreads the adds.
#pragma once

#include <cuda_runtime.h>

#include "ptx.cuh"

namespace fpo {

constexpr int kSlotBlocks = 8;     // blocks per cluster, and clusters per layer: 1
constexpr int kSlotThreads = 256;

__device__ __forceinline__ double ld_shared_cluster_f64(uint32_t cluster_addr) {
    double v;
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(cluster_addr) : "memory");
    return v;
}

// Totals of p[0, slots) (N floats each) in a fixed order: thread-strided sums, a butterfly
// per warp, the warps' sums in order, the blocks' sums in rank order.  Every thread of the
// cluster calls it; true in the one thread that holds the totals.
template <int N>
__device__ __forceinline__ bool slot_sum(const float* p, int slots, double (&tot)[N]) {
    __shared__ double warp_part[kSlotThreads / 32][N];
    __shared__ double block_part[N];
    const int rank = static_cast<int>(cluster_ctarank());
    double acc[N];
#pragma unroll
    for (int j = 0; j < N; ++j) acc[j] = 0.0;
#pragma unroll 4
    for (int i = rank * kSlotThreads + threadIdx.x; i < slots; i += kSlotBlocks * kSlotThreads) {
#pragma unroll
        for (int j = 0; j < N; ++j) acc[j] += p[static_cast<size_t>(i) * N + j];
    }
#pragma unroll
    for (int j = 0; j < N; ++j) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
        if ((threadIdx.x & 31) == 0) warp_part[threadIdx.x >> 5][j] = acc[j];
    }
    __syncthreads();
    if (threadIdx.x < N) {
        double t = 0.0;
        for (int w = 0; w < kSlotThreads / 32; ++w) t += warp_part[w][threadIdx.x];
        block_part[threadIdx.x] = t;
    }
    cluster_sync();
    const bool mine = rank == 0 && threadIdx.x == 0;
    if (mine) {
#pragma unroll
        for (int j = 0; j < N; ++j) {
            tot[j] = 0.0;
            for (int r = 0; r < kSlotBlocks; ++r)
                tot[j] += ld_shared_cluster_f64(
                    mapa_shared(smem_u32(&block_part[j]), static_cast<uint32_t>(r)));
        }
    }
    cluster_sync();  // no block leaves while its sums are read
    return mine;
}

}  // namespace fpo
