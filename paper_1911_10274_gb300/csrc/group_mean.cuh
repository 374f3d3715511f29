// group_mean.cuh -- mean position of groups of masses, in FP64 and in a fixed
// order (the swarm objective of both the single-system and the batch engine).
//
// Bound: the latency of the scattered state reads, and of FP64 sums (the device adds
// few FP64 numbers at a time).  A thread per group left a 1,728-mass robot as a chain
// of dependent loads and adds (814 us for 256 robots); 128 threads per group keep
// that many reads in flight and the sums are added pairwise: 256 robots' rollout and
// gradient 11.5 -> 10.8 ms, 1,024 robots' 200-step rollout with its centroids 6.66 ->
// 6.16 ms.  Small groups are better off with fewer threads: with launch and wait,
// 100,000 groups of 8 masses took 38 us by a thread each and 1,306 by a block each,
// 20,000 of 32 41 by a thread and 87 by a warp (15 sums across its lanes).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace titan {

constexpr int kMeanThreads = 128;

constexpr int kMeanFew = 8;

// Threads per group for n_groups groups of n masses in all: one for groups smaller than
// a warp on average, eight for groups smaller than a block, else a block.
constexpr uint32_t mean_lanes(uint64_t n, uint32_t n_groups) {
    return n < 32ull * n_groups ? 1 : n < (uint64_t)kMeanThreads * n_groups ? kMeanFew : kMeanThreads;
}
constexpr uint32_t mean_blocks(uint64_t n, uint32_t n_groups) {
    const uint32_t per = kMeanThreads / mean_lanes(n, n_groups);
    return n_groups / per + (n_groups % per != 0);
}

// s = load(first) + load(first + step) + ... below count, one thread's share.
template <typename Load>
__device__ __forceinline__ void strided_sum(uint32_t first, uint32_t step, uint32_t count, Load &load, double *s) {
    s[0] = s[1] = s[2] = 0;
#pragma unroll 4
    for (uint32_t i = first; i < count; i += step) {
        const float4 p = load(i);
        s[0] += p.x;
        s[1] += p.y;
        s[2] += p.z;
    }
}

// The sum of s over each LANES lanes of a warp (all of which call it), pairwise, in every lane.
template <int LANES>
__device__ __forceinline__ void lane_sum(double *s) {
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int o = LANES / 2; o; o >>= 1) s[a] += __shfl_xor_sync(0xffffffffu, s[a], o);
}

// One group by the whole block (which calls it): thread t adds masses t, t + 128, ...
// in turn, then the partial sums are added in a fixed tree.
template <typename Load, typename Store>
__device__ __forceinline__ void block_mean(uint32_t count, Load &load, Store &store) {
    __shared__ double part[3][kMeanThreads / 32];
    double s[3];
    strided_sum(threadIdx.x, kMeanThreads, count, load, s);
    lane_sum<32>(s);
    __syncthreads();                                        // the group before is done with `part`
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int a = 0; a < 3; ++a) part[a][threadIdx.x >> 5] = s[a];
    __syncthreads();
    if (threadIdx.x < 3) {
        double t = 0;
#pragma unroll
        for (int w = 0; w < kMeanThreads / 32; ++w) t += part[threadIdx.x][w];
        store(threadIdx.x, count ? t / (double)count : 0.0);
    }
}

// The groups of this block, LANES threads (mean_lanes) to each: group g < n_groups has
// count(g) masses at load(g, 0 ..) and gets store(g, axis, mean) once per axis, with 0
// if it is empty.  With fewer lanes than the block, groups of more masses than the
// block has threads are left to the whole block at the end.
template <int LANES, typename Count, typename Load, typename Store>
__device__ __forceinline__ void group_means(uint32_t n_groups, Count &&count, Load &&load, Store &&store) {
    constexpr uint32_t PER = kMeanThreads / LANES;
    const uint32_t g = blockIdx.x * PER + threadIdx.x / LANES;
    auto whole = [&](uint32_t group, uint32_t c) {
        auto at = [&](uint32_t i) { return load(group, i); };
        auto put = [&](uint32_t axis, double m) { store(group, axis, m); };
        block_mean(c, at, put);
    };
    if constexpr (LANES == kMeanThreads) {
        whole(g, count(g));
    } else {
        __shared__ uint32_t counts[PER];
        const uint32_t c = g < n_groups ? count(g) : 0;
        const bool large = c > (uint32_t)kMeanThreads;
        if (threadIdx.x % LANES == 0) counts[threadIdx.x / LANES] = c;
        auto at = [&](uint32_t i) { return load(g, i); };
        double s[3];
        strided_sum(threadIdx.x % LANES, LANES, large ? 0 : c, at, s);
        lane_sum<LANES>(s);
        if (threadIdx.x % LANES == 0 && !large && g < n_groups) {
            const double inv = c ? 1.0 / (double)c : 0.0;   // one FP64 division, not three
#pragma unroll
            for (int a = 0; a < 3; ++a) store(g, a, s[a] * inv);
        }
        if (!__syncthreads_or(large)) return;
        for (uint32_t k = 0; k < PER; ++k)
            if (counts[k] > (uint32_t)kMeanThreads) whole(blockIdx.x * PER + k, counts[k]);
    }
}

}  // namespace titan
