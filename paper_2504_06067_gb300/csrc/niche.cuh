// niche.cuh -- Philox priorities and the block scan of the niche selection,
// shared by its kernels (k_niche.cu) and the one-cluster generation
// (k_small.cu).
#pragma once
#include "common.cuh"

namespace {

__device__ __forceinline__ uint32_t mem_prio(uint64_t seed, uint32_t gen, int i)
{
    return philox((uint32_t)i, gen, RNG_MEMPRIO, 0u, seed).x;
}

__device__ __forceinline__ unsigned long long ref_key(uint64_t seed, uint32_t gen, int j)
{
    return ((unsigned long long)philox((uint32_t)j, gen, RNG_REFPRIO, 0u, seed).x << 32) | (unsigned)j;
}

// exclusive scan of one value per thread; returns the prefix, *total the sum
__device__ int block_excl_scan(int x, int* scratch, int* total)
{
    const int lane = lane_id(), warp = threadIdx.x >> 5;
    int inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) scratch[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int v = (lane < (int)(blockDim.x >> 5)) ? scratch[lane] : 0;
        int vi = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, vi, o);
            if (lane >= o) vi += y;
        }
        scratch[lane] = vi - v;
        if (lane == 31) scratch[32] = vi;
    }
    __syncthreads();
    const int res = scratch[warp] + inc - x;
    *total = scratch[32];
    __syncthreads();
    return res;
}

}  // namespace
