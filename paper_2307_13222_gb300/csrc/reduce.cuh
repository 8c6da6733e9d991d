// Sum of per-block partials by one thread block.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace hphi {

constexpr int kSumThreads = 128;  // threads of the partial-sum kernels

// Sum of p[0], p[stride], ..., p[(n - 1) stride] over the thread block
// (kSumThreads threads, all of them call): thread t adds t, t + kSumThreads, ...
// in order, then a fixed butterfly and the warps in order, so a result depends
// on n alone.  The total is valid in thread 0.  (A launch has up to 1216
// partials per value: one thread adding them one by one took 26 to 110 us, the
// latency of 1216 dependent FP64 adds; this takes about 3.)
static __device__ __forceinline__ double block_sum_strided(const double *__restrict__ p, int n, int64_t stride) {
    __shared__ double sm[kSumThreads / 32];
    double s = 0.0;
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += kSumThreads) s += p[i * stride];
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = s;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
#pragma unroll
        for (int w = 0; w < kSumThreads / 32; w++) t += sm[w];
    return t;
}

}  // namespace hphi
