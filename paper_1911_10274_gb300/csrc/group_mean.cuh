// group_mean.cuh -- mean position of one group of masses by one block, in FP64
// and in a fixed order (the swarm objective of both the single-system and the
// batch engine).
//
// Bound: the latency of the scattered state reads.  One thread per group left
// a 1,728-mass robot as a chain of dependent loads and FP64 adds (814 us for
// 256 robots); 128 threads per group keep that many reads in flight and the
// sums are added pairwise: 256 robots' rollout and gradient 11.5 -> 10.8 ms, 1,024
// robots' 200-step rollout with its centroids 6.66 -> 6.16 ms.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace titan {

constexpr int kMeanThreads = 128;

// m = the mean of load(0) .. load(count - 1) (x, y, z of a float4); 0 for an
// empty group.  Thread t adds masses t, t + kMeanThreads, ... in turn, then the
// partial sums are added in a fixed tree.  Every thread of the block calls it;
// the result is valid in every thread.
template <typename Load>
__device__ __forceinline__ void group_mean(uint32_t count, Load load, double *m) {
    __shared__ double part[3][kMeanThreads / 32];
    double s[3] = {0, 0, 0};
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < count; i += kMeanThreads) {
        const float4 p = load(i);
        s[0] += p.x;
        s[1] += p.y;
        s[2] += p.z;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        for (int o = 16; o; o >>= 1) s[a] += __shfl_xor_sync(0xffffffffu, s[a], o);
        if ((threadIdx.x & 31) == 0) part[a][threadIdx.x >> 5] = s[a];
    }
    __syncthreads();
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double t = 0;
#pragma unroll
        for (int w = 0; w < kMeanThreads / 32; ++w) t += part[a][w];
        m[a] = count ? t / (double)count : 0.0;
    }
}

}  // namespace titan
