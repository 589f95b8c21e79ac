// dot_reduce.cuh -- block and grid sums of the stopping measures (both precisions).
//
// A 32-lane FP64 addition occupies an SM for 16 cycles: a block adds up only the sums of
// its kind, and a warp's tree halves the number of sums a lane carries at every exchange
// (16 additions for 16 sums instead of 80).
#pragma once
#include <cuda_runtime.h>

#include "dot_internal.cuh"

namespace dot {

// Sums of v[0 .. 15] over the warp: lane l returns the sum of v[l / 2].
__device__ __forceinline__ double warp_sums16(double* v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int h = 8; h >= 1; h /= 2) {   // lanes exchange at distance 2 h and keep half of their sums
    const bool up = lane & (2 * h);
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const double send = up ? v[k] : v[k + h], keep = up ? v[k + h] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * h);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// Block sums of the slots listed in `which` into column `row` of out[R_NSLOTS][rows]; the
// other slots' entries are zero.
template <int THREADS, int NS>
__device__ __forceinline__ void block_reduce_store(const double (&val)[NS], const int (&which)[NS], double* out,
                                                   int rows, int row) {
  static_assert(NS <= 16, "one exchange tree");
  __shared__ double sh[THREADS / 32][16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) v[k] = k < NS ? val[k < NS ? k : 0] : 0.0;
  const double t = warp_sums16(v);
  if ((lane & 1) == 0) sh[warp][lane >> 1] = t;
  __syncthreads();
  if (threadIdx.x < R_NSLOTS) {
    int at = -1;
#pragma unroll
    for (int k = 0; k < NS; ++k)
      if (which[k] == (int)threadIdx.x) at = k;
    double s = 0.0;
    if (at >= 0)
      for (int w = 0; w < THREADS / 32; ++w) s += sh[w][at];
    out[(long long)threadIdx.x * rows + row] = s;
  }
}

// The sum of p[0 .. rows) by a block of 128 threads, in a fixed order; thread 0 returns it.
__device__ __forceinline__ double row_sum128(const double* p, int rows) {
  double v = 0.0;
#pragma unroll 4
  for (int r = threadIdx.x; r < rows; r += 128) v += p[r];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __shared__ double sh[4];
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  return (sh[0] + sh[1]) + (sh[2] + sh[3]);
}

}  // namespace dot
