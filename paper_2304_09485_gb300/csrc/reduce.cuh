// Reductions with a fixed order of summation.
#pragma once
#include <cuda_runtime.h>

namespace hgks {

// Whether a counter of arrivals has reached `want`. Both are taken modulo 2^32: a solve of many
// restarts passes 2^32 arrivals (28 million barriers of 152 blocks), and the counter is never
// further than one barrier's blocks from what is waited for.
__host__ __device__ inline bool arrived(unsigned seen, unsigned want) { return (int)(seen - want) >= 0; }

// The sums over a warp of K values per lane (K a power of two): lane l returns the sum of
// value l / (32 / K). Each exchange halves the values a lane holds, so the K sums take
// K - 1 + log2(32 / K) additions instead of 5 K: a warp-wide FP64 addition holds
// the SM's FP64 pipe for 16 clocks.
template <int K>
__device__ __forceinline__ double warp_sums(double *v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = K / 2, o = 16; s >= 1; s >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int q = 0; q < s; q++) {
      const double send = up ? v[q] : v[q + s], keep = up ? v[q + s] : v[q];
      v[q] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  double t = v[0];
#pragma unroll
  for (int o = 16 / K; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// The sums over a block of K values per thread, in sh[0][k] (after a __syncthreads):
// warps first, then the warps in order. sh: [warps][K].
template <int K, int WARPS>
__device__ __forceinline__ void block_sums(double *v, double (*sh)[K]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double t = warp_sums<K>(v);
  if (lane % (32 / K) == 0) sh[warp][lane / (32 / K)] = t;
  __syncthreads();
  if (threadIdx.x < K) {
    double s = sh[0][threadIdx.x];
#pragma unroll
    for (int w = 1; w < WARPS; w++) s += sh[w][threadIdx.x];
    sh[0][threadIdx.x] = s;
  }
  __syncthreads();
}

}  // namespace hgks
