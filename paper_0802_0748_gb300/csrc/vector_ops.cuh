// Deterministic reductions of the standalone vector kernels (256-thread
// blocks) of the ground-state iteration.
#pragma once
#include "common.cuh"

namespace scocg {

// Reductions of 256-thread blocks: a block's partial sum lands in
// part[blockIdx.x], and the G partials are added in one fixed order.  Separate
// launches have the last block of the producing one add them (block_total); the
// cooperative recursion and the projections add them where they are used
// (sum_partials): every block that does sees the same bits.
constexpr int kVecBlock = 256;

__device__ __forceinline__ void block_partial(double v, double* part) {
    __shared__ double s_w[kVecBlock / 32];
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kVecBlock / 32; ++w) t += s_w[w];
        part[blockIdx.x] = t;
    }
}

__device__ __forceinline__ double sum_partials(const double* part, int G) {
    __shared__ double s_w[kVecBlock / 32];
    __shared__ double s_tot;
    double v = 0.0;
    for (int c = threadIdx.x; c < G; c += kVecBlock) v += __ldcg(part + c);
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kVecBlock / 32; ++w) t += s_w[w];
        s_tot = t;
    }
    __syncthreads();
    return s_tot;
}

// The same with the sum of all blocks' partials: the block that arrives last adds
// them (in sum_partials' order) and stores the total, so that a consuming launch
// reads one number; summed by every consuming block the partials cost a vector
// pass of 853,776 rows ~8 of its 17 us (an FP64 instruction holds the SM's pipe 16
// cycles, and 64 warps of an SM repeated it).  `part` is preceded by kPartHead
// doubles, {total, arrival count}, zeroed once before the first launch.  True in
// the last block, after the total is stored.
constexpr int kPartHead = 2;
__device__ __forceinline__ double total_of(const double* part) { return __ldcg(part - kPartHead); }
__device__ __forceinline__ bool block_total(double v, double* part) {
    __shared__ int s_last;
    block_partial(v, part);
    if (threadIdx.x == 0) {
        __threadfence();
        unsigned* count = reinterpret_cast<unsigned*>(part - 1);
        s_last = atomicInc(count, gridDim.x - 1) == gridDim.x - 1;   // wraps to 0 for the next launch
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return false;
    const double s = sum_partials(part, (int)gridDim.x);
    if (threadIdx.x == 0) part[-kPartHead] = s;
    return true;
}

}  // namespace scocg
