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

// x rounded to a multiple of 2^(emax - 1076), in these units (emax: the largest exponent field
// among the values summed): at most 2^54, and at most 320 of them.
__device__ __forceinline__ long long gram_fixed(double x, int emax) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  const long long m = ((b & 0xfffffffffffffLL) | (e ? 1LL << 52 : 0)) << 1;
  const int sh = emax - max(e, 1);
  const long long q = sh > 55 ? 0 : (m + ((1LL << sh) >> 1)) >> sh;
  return b < 0 ? -q : q;
}
// and back; NaN when a value summed was not finite (the factorisation then reports a breakdown)
__device__ __forceinline__ double gram_float(long long s, int emax) {
  if (emax == 0x7ff) return __longlong_as_double(0x7ff8000000000000LL);
  return emax > 53 ? (double)s * __hiloint2double((emax - 53) << 20, 0) : ldexp((double)s, emax - 1076);
}

// G[e] = sum of the nparts <= gram_sum_most(nn) partials of entry e ([entry][part]), order-
// independent; 256 threads, ends with a barrier.  The partials are added as integers on the
// largest one's scale, real and imaginary parts each on their own: an FP64 add holds the FP64
// unit for 64 cycles, and 28 of them in turn took 1.8 us of the coefficient step's 9 at n = 4.
// Rounding is to 2^-53 of the largest partial per partial, which is no coarser than the adds'.
__device__ __forceinline__ void gram_sum_parts(double2 *G, const double2 *__restrict__ part, int nparts, int nn) {
  const int T = gram_sum_lanes(nn);
  const int e = threadIdx.x / T, q = threadIdx.x - e * T;
  if (nparts == 1) {
    if (e < nn && q == 0) G[e] = part[e];
    __syncthreads();
    return;
  }
  double2 v[10];
  int ex = 1, ey = 1;
#pragma unroll
  for (int u = 0; u < 10; ++u) {
    const int p = q + u * T;
    v[u] = (e < nn && p < nparts) ? part[(long)e * nparts + p] : make_double2(0.0, 0.0);
  }
#pragma unroll
  for (int u = 0; u < 10; ++u) {
    ex = max(ex, (__double2hiint(v[u].x) >> 20) & 0x7ff);
    ey = max(ey, (__double2hiint(v[u].y) >> 20) & 0x7ff);
  }
  for (int off = T / 2; off > 0; off >>= 1) {  // (T divides 32: the lanes of an entry share a warp)
    ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, off));
    ey = max(ey, __shfl_xor_sync(0xffffffffu, ey, off));
  }
  long long sx = 0, sy = 0;
#pragma unroll
  for (int u = 0; u < 10; ++u) {
    sx += gram_fixed(v[u].x, ex);
    sy += gram_fixed(v[u].y, ey);
  }
  for (int off = T / 2; off > 0; off >>= 1) {
    sx += __shfl_xor_sync(0xffffffffu, sx, off);
    sy += __shfl_xor_sync(0xffffffffu, sy, off);
  }
  if (T > 1) {  // lanes 0 and 1 of an entry convert one component each
    if (e < nn && q < 2) reinterpret_cast<double *>(G)[2 * e + q] = gram_float(q ? sy : sx, q ? ey : ex);
  } else if (e < nn) {
    G[e] = make_double2(gram_float(sx, ex), gram_float(sy, ey));
  }
  __syncthreads();
}

}  // namespace rhmc
