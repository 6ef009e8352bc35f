// Sums of per-CTA partials, in a fixed order.
//
// The producers leave up to 1216 partials for every output (8 CTAs per SM),
// an array parts[nparts][count] with the outputs fastest.  A single thread
// that walks 1216 partials waits for 1216 loads one after the other, and the
// FP64 adds of a warp take 64 cycles each, so the work has to be spread over
// the chip: a CTA takes C consecutive outputs (C * sizeof(T) >= one 32-byte
// sector) and R threads per output, thread (r, c) adds parts r, r + R, ...;
// the R sums are then added pairwise in shared memory.
#pragma once
#include "common.cuh"

__device__ __forceinline__ void acc_add(double &a, double b) { a += b; }
__device__ __forceinline__ void acc_add(cxd &a, cxd b) { a = a + b; }
__device__ __forceinline__ void acc_zero(double &a) { a = 0.0; }
__device__ __forceinline__ void acc_zero(cxd &a) { a = mk(0.0, 0.0); }

// Sum of column `col` of parts (row length `count`, valid when ok); the CTA
// has C * R threads, thread r * C + c works on the CTA's column c.  sm: C * R
// entries.  The result is returned in the threads with r == 0.
template <int C, int R, typename T>
__device__ __forceinline__ T column_sum(const T *__restrict__ parts, int nparts, size_t count, size_t col, bool ok,
                                        T *sm) {
  const int r = threadIdx.x / C;
  T s0, s1;
  acc_zero(s0);
  acc_zero(s1);
  if (ok) {
    int p = r;
    for (; p + 3 * R < nparts; p += 4 * R) {
      T v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = parts[(size_t)(p + u * R) * count + col];
      acc_add(v[0], v[1]);
      acc_add(v[2], v[3]);
      acc_add(s0, v[0]);
      acc_add(s1, v[2]);
    }
    for (; p < nparts; p += R) acc_add(s0, parts[(size_t)p * count + col]);
  }
  acc_add(s0, s1);
  sm[threadIdx.x] = s0;
  __syncthreads();
#pragma unroll
  for (int o = R / 2; o > 0; o >>= 1) {
    if (r < o) {
      acc_add(s0, sm[threadIdx.x + o * C]);
      sm[threadIdx.x] = s0;
    }
    __syncthreads();
  }
  return s0;
}
