// Sums over the blocks of a launch without a second one.
#pragma once

#include "field_fast.cuh"
#include "running_sum.h"

namespace jdft {

// Sum over the block in a fixed order; thread 0 returns it.
template <int THREADS>
__device__ __forceinline__ double block_total(double x) {
    __shared__ double red[THREADS / 32];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int i = 0; i < THREADS / 32; ++i) s += red[i];
    return s;
}

// out[k] = scale * sum over blocks of x[k], k < NOUT: the block's sums go to
// partial[NOUT * block + k]; the last block to arrive adds them, each thread its
// share of the blocks in order, then the threads in order (deterministic), and
// resets the counter for the next launch.
template <int NOUT, int THREADS>
__device__ __forceinline__ void finish_sum(const double* x, const BlockSum& b, double scale) {
    __shared__ bool last;
#pragma unroll
    for (int k = 0; k < NOUT; ++k) {
        const double s = block_total<THREADS>(x[k]);
        if (threadIdx.x == 0) b.partial[NOUT * blockIdx.x + k] = s;
    }
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(b.count, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int k = 0; k < NOUT; ++k) {
        double t = 0.0;
        for (int i = threadIdx.x; i < (int)gridDim.x; i += THREADS) t += __ldcg(&b.partial[NOUT * i + k]);
        t = block_total<THREADS>(t);
        if (threadIdx.x == 0) b.out[k] = scale * t;
    }
    if (threadIdx.x == 0) *b.count = 0u;
}

}  // namespace jdft
