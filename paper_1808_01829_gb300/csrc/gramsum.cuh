// Sum of a Gram matrix's per-CTA partials inside the n x n kernels: on small lattices the
// separate summing kernel (2 to 3 us, one CTA per entry) costs more than the sum.
#pragma once

#include "common.cuh"

namespace rhmc {

// Lanes per entry: the largest power of two with lanes x n^2 <= 256, at most 32.
__host__ __device__ __forceinline__ int gram_sum_lanes(int nn) {
  int t = 1;
  while (t < 32 && 2 * t * nn <= 256) t *= 2;
  return t;
}
// Up to this many partials the n x n kernel sums them itself (ten loads per lane, about
// 1.5 us of FP64 adds; 256 entries of 8 partials at n = 16)
__host__ __device__ __forceinline__ int gram_sum_most(int nn) { return 10 * gram_sum_lanes(nn); }

// G[e] = sum of the nparts partials of entry e ([entry][part]), fixed order; 256 threads, ends
// with a barrier.
__device__ __forceinline__ void gram_sum_parts(double2 *G, const double2 *__restrict__ part, int nparts, int nn) {
  const int T = gram_sum_lanes(nn);
  const int e = threadIdx.x / T, q = threadIdx.x - e * T;
  double2 s = make_double2(0.0, 0.0);
  if (e < nn) {
#pragma unroll 5
    for (int p = q; p < nparts; p += T) {
      const double2 v = part[(long)e * nparts + p];
      s.x += v.x;
      s.y += v.y;
    }
  }
  for (int off = T / 2; off > 0; off >>= 1) {  // (T divides 32: the lanes of an entry share a warp)
    s.x += __shfl_xor_sync(0xffffffffu, s.x, off);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, off);
  }
  if (e < nn && q == 0) G[e] = s;
  __syncthreads();
}

}  // namespace rhmc
