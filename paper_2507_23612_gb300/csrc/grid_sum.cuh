// Sum over a grid in one launch.
#pragma once
#include <cuda_runtime.h>

namespace hub {

// The sum of one double per thread of the grid, in the CTA that comes last (true for its thread 0):
// no launch of its own for the second stage, and a fixed order (a CTA's warps, then the CTAs by
// index).  part: one double per CTA; the counter starts at zero and is left there.  All threads of a
// CTA (a multiple of 32, at most 1024) call it.
__device__ __forceinline__ bool grid_sum(double v, double* part, unsigned* counter, double& total) {
    __shared__ double red[32];
    __shared__ int last;
    const int warps = blockDim.x >> 5;
    auto block = [&](double t) {
        for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
        __syncthreads();
    };
    block(v);
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < warps; ++w) t += red[w];
        part[blockIdx.x] = t;
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
        if (last) *counter = 0;
        __threadfence();
    }
    __syncthreads();
    if (!last) return false;
    double t = 0.0;
#pragma unroll 4
    for (unsigned i = threadIdx.x; i < gridDim.x; i += blockDim.x) t += __ldcg(part + i);
    block(t);
    total = 0.0;
    for (int w = 0; w < warps; ++w) total += red[w];
    return threadIdx.x == 0;
}

}  // namespace hub
