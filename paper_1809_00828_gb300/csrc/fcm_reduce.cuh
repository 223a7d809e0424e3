// Deterministic sums over a grid (internal to libfcm): warp shuffles, one partial per CTA, and the last CTA to
// finish (ticket counter) adds the partials in a fixed order.
//
// What bounds them at the sizes of a solve is the latency of the chain of FP64 additions (and, with many CTAs per
// SM, the FP64 pipe: 2 operations per clock per SM), so several sums go through the rounds together, the second
// stage takes the 3 rounds that 8 warps need, and no sum is carried that nobody reads (32^3 cells, coarse CG: the
// product of K_H 28.2 -> 25.6 us, the update 8.7 -> 7.2; a flexible solve of 172 iterations 178 -> 164 ms).
#pragma once

#include <cuda_runtime.h>

namespace fcm {

constexpr int kReduceThreads = 256, kReduceWarps = kReduceThreads / 32;

// Sums of v[k] over the CTA's first `warps` warps (the others hold nothing); valid in thread 0.
template <int N>
__device__ __forceinline__ void block_sums(double (&v)[N], double (*sh)[kReduceWarps], int warps = kReduceWarps)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < warps) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < N; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
        if (lane == 0)
#pragma unroll
            for (int k = 0; k < N; ++k) sh[k][warp] = v[k];
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] = lane < warps ? sh[k][lane] : 0.0;
#pragma unroll
        for (int o = kReduceWarps / 2; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < N; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    }
}

// Sums of v[k] over the grid; true in the last CTA, whose thread 0 then holds them.  `partial`: N doubles per CTA.
template <int N>
__device__ __forceinline__ bool grid_sums(double (&v)[N], double *partial, unsigned *counter, int warps = kReduceWarps)
{
    __shared__ double sh[N][kReduceWarps];
    __shared__ bool last;
    block_sums(v, sh, warps);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) partial[N * blockIdx.x + k] = v[k];
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return false;
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += kReduceThreads)
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] += __ldcg(partial + N * i + k);
    block_sums(v, sh);
    if (threadIdx.x == 0) *counter = 0u;
    return true;
}

}  // namespace fcm
