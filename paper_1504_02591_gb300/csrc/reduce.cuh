// reduce.cuh: the fixed-order float64 sums of per-block partials.
#pragma once
#include <cuda_runtime.h>

namespace rg {

// float64 adds run at 2 a clock and SM, so the sum is bound by them and by the latency of its steps, not by
// its bytes: 256 threads keep the adds of the trees few (1024 threads spent 2.5 us in them alone), and
// beyond 1024 partials more blocks share the work.
constexpr int kReduceThreads = 256;

inline int reduce_blocks(int nblocks, int most) {
  const int b = (nblocks + 1023) / 1024;
  return b < 1 ? 1 : (b > most ? most : b);
}

// Sum nq <= 4 interleaved columns of nblocks partials in a fixed order, by kReduceThreads threads a block.
// Several blocks (at most 64) each sum a contiguous range, leave it in bsum (4 doubles a block), and the
// last one to finish adds the blocks' sums and resets the counter.  True in the one thread that holds the
// sums.
__device__ __forceinline__ bool reduce_partials(const double* __restrict__ partials, int nblocks, int nq,
                                                double* __restrict__ bsum, unsigned int* __restrict__ counter,
                                                double (&t)[4]) {
  constexpr int W = kReduceThreads / 32;
  __shared__ double sh[4][W];
  __shared__ bool last;
  const int per = (nblocks + gridDim.x - 1) / gridDim.x;
  const int b0 = blockIdx.x * per, b1 = min(nblocks, b0 + per);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < 4; ++q) t[q] = 0.0;
#pragma unroll 4
  for (int b = b0 + threadIdx.x; b < b1; b += kReduceThreads)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < nq) t[q] += partials[(size_t)b * nq + q];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (q < nq) {
      for (int o = 16; o > 0; o >>= 1) t[q] += __shfl_down_sync(0xffffffffu, t[q], o);
      if (l == 0) sh[q][w] = t[q];
    }
  __syncthreads();
  if (w == 0)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < nq) {
        t[q] = l < W ? sh[q][l] : 0.0;
        for (int o = W / 2; o > 0; o >>= 1) t[q] += __shfl_down_sync(0xffffffffu, t[q], o);
      }
  if (gridDim.x == 1) return threadIdx.x == 0;
  if (threadIdx.x == 0) {
    for (int q = 0; q < nq; ++q) bsum[4 * blockIdx.x + q] = t[q];
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last || w != 0) return false;
  __threadfence();
  const volatile double* vb = bsum;
  const int g = (int)gridDim.x;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (q < nq) {
      t[q] = l < g ? vb[4 * l + q] : 0.0;
      if (l + 32 < g) t[q] += vb[4 * (l + 32) + q];
      for (int o = 16; o > 0; o >>= 1) t[q] += __shfl_down_sync(0xffffffffu, t[q], o);
    }
  if (l == 0) *counter = 0u;
  return l == 0;
}

}  // namespace rg
