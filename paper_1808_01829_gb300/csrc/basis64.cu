// FP64 solve with the stored block Krylov basis.
//
// The shifted updates of Algorithm 1 cost two n x n products per row, shift and
// iteration, at this GPU's FP64 rate the largest part of an FP64 solve (36 us on average
// per update at 8^4, n = 4, 11 shifts, against 100 us per iteration).  As in the
// mixed solve (basis.cu), the solve keeps the blocks Q_0, Q_1, ... and the recorded
// n x n coefficients, and forms the shifted solutions once at the end,
//   X^(s) = sum_{i < L_s} Q_i C^(s)_i,
// one product per row, shift and iteration instead of two, off the iteration's path,
// without P^(s) and X^(s) going through memory.  Where only the rational sum
// sum_s w_s X^(s) is wanted (heatbath, action), the coefficients are summed first:
// one product per row and iteration for all shifts together.
// The blocks are written where they stay (a table of blocks [rows][n], so that a solve takes memory as
// it goes): iteration k forms Q_k in block k of the basis (k from the device counter: graph replays).
#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "fx.cuh"
#include "kernels.h"

namespace rhmc {

namespace {
// Rows of n columns, one lane per (row, column); the rows of a warp lie side by side and do
// not straddle it (32 / N rows, the remaining lanes idle).
template <int N> struct Lanes {
  static constexpr int RPW = 32 / N;
  long row;
  int j;
  bool in;
  __device__ Lanes(long base, long rows) {
    const int lane = threadIdx.x & 31, slot = lane / N;
    j = lane - slot * N;
    row = base + (threadIdx.x >> 5) * RPW + slot;
    in = slot < RPW && row < rows;
  }
};
}  // namespace

// W = Q_{k-1} + A M: the block QR step, Q_{k-1} in block *kdev - 1 of the basis.  One lane per
// output, so that small lattices spread over the FP64 units of the whole GPU (each FP64
// instruction of a warp takes 64 clocks however few there are).
template <int N>
__global__ void __launch_bounds__(128) k_axpy64(const double2 *__restrict__ A, double2 *const *__restrict__ basis,
                                                const int *__restrict__ kdev, const double2 *__restrict__ M,
                                                double2 *__restrict__ Y, long rows) {
  __shared__ double2 sm[N * N];
  for (int k = threadIdx.x; k < N * N; k += blockDim.x) sm[k] = M[k];
  const double2 *Q = basis[*kdev - 1];
  __syncthreads();
  const long per = 4 * Lanes<N>::RPW;
  for (long base = (long)blockIdx.x * per; base < rows; base += (long)gridDim.x * per) {
    const Lanes<N> l(base, rows);
    if (!l.in) continue;
    double2 acc = czero<double>();
#pragma unroll
    for (int k = 0; k < N; ++k) cmac<double>(acc, __ldg(A + l.row * N + k), sm[k * N + l.j]);
    const double2 q = Q[l.row * N + l.j];
    Y[l.row * N + l.j] = make_double2(q.x + acc.x, q.y + acc.y);
  }
}

// The base updates of Algorithm 1 after rho_k: Q_k = W rho^-1 into block *kdev of the basis,
// X^(0) += P M1, P = Q_k + P M2.  rho^-1 is upper and M2 = rho^dagger lower triangular, so
// column j of Q takes terms k <= j and column j of P M2 terms k >= j: n + 1 products
// together, formed in one running sum whose value after the first j + 1 is Q.
template <int N>
__global__ void __launch_bounds__(128) k_base64(const double2 *__restrict__ W, double2 *const *__restrict__ basis,
                                                const int *__restrict__ kdev, double2 *P, double2 *X,
                                                const double2 *__restrict__ coef, long rows) {
  __shared__ double2 sm[3 * N * N];
  for (int k = threadIdx.x; k < 3 * N * N; k += blockDim.x) sm[k] = coef[k];
  double2 *Q = basis[*kdev];
  __syncthreads();
  const long per = 4 * Lanes<N>::RPW;
  for (long base = (long)blockIdx.x * per; base < rows; base += (long)gridDim.x * per) {
    const Lanes<N> l(base, rows);
    double2 p[N];
    const long o = l.row * N;
    if (l.in) {
#pragma unroll
      for (int k = 0; k < N; ++k) p[k] = P[o + k];
    }
    __syncwarp();  // the row is read by all its lanes before any of them writes its column
    if (l.in) {
      double2 x = X[o + l.j], a = czero<double>(), q = czero<double>(), acc = czero<double>();
#pragma unroll
      for (int t = 0; t <= N; ++t) {
        if (t == l.j + 1) q = acc;
        const bool first = t <= l.j;
        const double2 u = first ? __ldg(W + o + (t < N ? t : N - 1)) : p[t > 0 ? t - 1 : 0];
        const double2 c = first ? sm[(t < N ? t : N - 1) * N + l.j] : sm[2 * N * N + (t > 0 ? t - 1 : 0) * N + l.j];
        cmac<double>(acc, u, c);
      }
#pragma unroll
      for (int k = 0; k < N; ++k) cmac<double>(a, p[k], sm[N * N + k * N + l.j]);
      Q[o + l.j] = q;
      P[o + l.j] = acc;
      X[o + l.j] = make_double2(x.x + a.x, x.y + a.y);
    }
    __syncwarp();
  }
}

// Weighted sum of the shifts' expansion coefficients (basis_coef's cf): block i of the sum
// takes w_s C^(s)_i of every shift s >= 1 with more than i blocks.
__global__ void __launch_bounds__(256) k_basis64_combine(int n, int nshift, const SolverState *__restrict__ st, int K,
                                                         const double2 *__restrict__ cf, long cfstride,
                                                         double2 *__restrict__ out) {
  const int i = blockIdx.x, t = threadIdx.x, nn = n * n;
  if (t >= nn) return;
  double2 sum = make_double2(0.0, 0.0);
  for (int s = 1; s < nshift; ++s) {
    if (i >= min(st->last_k[s], K)) continue;
    const double w = st->w1[s];
    const double2 c = cf[((size_t)(s - 1) * cfstride + i) * nn + t];
    sum.x = fma(w, c.x, sum.x);
    sum.y = fma(w, c.y, sum.y);
  }
  out[(size_t)i * nn + t] = sum;
}

constexpr int kFar = 6;  // far below: 2^-kFar (2^-4 sends enough ordinary sums to the size loop to cost 471 us)
// sum_{i < nb, t < N} Q_{b + i}[row][t] C_i[t][j] in FP64
template <int N>
__device__ __noinline__ double2 basis64_terms(double2 *const *basis, int b, int nb, long row, int j,
                                              const double2 *cf) {
  double2 acc = czero<double>();
#pragma unroll 1
  for (int i = 0; i < nb; ++i)
#pragma unroll 1
    for (int t = 0; t < N; ++t) cmac<double>(acc, basis[b + i][row * N + t], cf[(i * N + t) * N + j]);
  return acc;
}

// out_s = sum_i Q_i C^(s)_i for the shifts s0 + SG blockIdx.y ... (want = 0: X^(s), last_s
// blocks; 1: P^(s), K + 1 blocks, active shifts; 2: one combined set, all K blocks).  One lane
// per (row, column), SG shifts each, so that a row of Q is read once for SG shifts.
// The products are exact integer sums (fx.cuh) over T blocks at a time, up to 24 terms: the
// row's entries in these blocks are brought to one exponent, as are the T n coefficients of
// each (shift, column), and a sum is added to the FP64 result as one value.  A term costs 9
// multiply-adds of four clocks where FP64 takes 4 of 64; converting and the FP64 value per
// sum take about as long again.  8^4, n = 4, 12 shifts: 379 us, 1250 us with FP64 FMAs.
// The error is 2^-55 of the largest entry times the largest coefficient; where the sum is far
// below that and so is the sum of the terms' sizes (columns that hardly mix, under weak links:
// large entries meet small coefficients), the terms are added in FP64 instead (small components
// of 1e-6: error 1.0e-10 -> 9.9e-14 of them; without the test 339 us).
// A block with an infinity or NaN gives NaN.
template <int N, int SG>
__global__ void __launch_bounds__(128, 4)
    k_basis64_apply(double2 *const *__restrict__ basis, long rows, const SolverState *__restrict__ st, int K, int want,
                    int nshift, const double2 *__restrict__ cf, long cfstride, double2 *__restrict__ out,
                    long fstride) {
  constexpr int NN = N * N, RPW = Lanes<N>::RPW;
  constexpr int T = 24 / N > 8 ? 8 : 24 / N < 1 ? 1 : 24 / N;  // blocks per sum
  __shared__ int4 sq[4][RPW * T * N];                         // rows: [slot][block][column]
  __shared__ int4 sc[SG * T * NN];                             // coefficients: [shift][block][row][column]
  __shared__ int ce[SG * N];                                   // largest exponent field of (shift, column)
  const int s0 = 1 + SG * blockIdx.y;
  int nblk[SG], most = 0;
#pragma unroll
  for (int g = 0; g < SG; ++g) {
    const int s = s0 + g;
    nblk[g] = s >= nshift ? 0 : want == 2 ? K : want == 1 ? (st->active[s] ? K + 1 : 0) : max(0, min(st->last_k[s], K));
    most = max(most, nblk[g]);
  }
  const Lanes<N> l((long)blockIdx.x * 4 * RPW, rows);
  const int lane = threadIdx.x & 31, slot = lane / N;
  int4 *wq = sq[threadIdx.x >> 5];
  double2 acc[SG];
#pragma unroll
  for (int g = 0; g < SG; ++g) acc[g] = czero<double>();
  for (int b = 0; b < most; b += T) {
    const int nb = min(T, most - b);
    // this lane's column of the row in the nb blocks, and the row's largest exponent field
    double2 v[T];
    int ef = 0;
#pragma unroll
    for (int i = 0; i < T; ++i) {
      v[i] = (l.in && i < nb) ? basis[b + i][l.row * N + l.j] : make_double2(0.0, 0.0);
      ef = max(ef, max(fx::expo(v[i].x), fx::expo(v[i].y)));
    }
    {
      const int own = ef;
#pragma unroll
      for (int q = 1; q < N; ++q) ef = max(ef, __shfl_sync(0xffffffffu, own, (slot * N + (l.j + q) % N) & 31));
    }
    __syncthreads();  // the previous sums have been formed
    for (int k = threadIdx.x; k < SG * N; k += blockDim.x) ce[k] = 0;
    if (slot < RPW) {
#pragma unroll
      for (int i = 0; i < T; ++i) {
        const int2 re = fx::split(v[i].x, ef), im = fx::split(v[i].y, ef);
        wq[(slot * T + i) * N + l.j] = make_int4(re.x, re.y, im.x, im.y);
      }
    }
    __syncthreads();
    double2 *raw = reinterpret_cast<double2 *>(sc);
    for (int k = threadIdx.x; k < SG * nb * NN; k += blockDim.x) {
      const int g = k / (nb * NN), r = k - g * (nb * NN), i = b + r / NN;
      int most_g = 0;
#pragma unroll
      for (int q = 0; q < SG; ++q) most_g = q == g ? nblk[q] : most_g;
      const double2 c = i < most_g ? cf[((size_t)(s0 - 1 + g) * cfstride + b) * NN + r] : make_double2(0.0, 0.0);
      raw[g * T * NN + r] = c;
      atomicMax(&ce[g * N + r % N], max(fx::expo(c.x), fx::expo(c.y)));
    }
    __syncthreads();
    for (int k = threadIdx.x; k < SG * nb * NN; k += blockDim.x) {
      const int g = k / (nb * NN), r = k - g * (nb * NN);
      const double2 c = raw[g * T * NN + r];
      const int e = ce[g * N + r % N];
      const int2 re = fx::split(c.x, e), im = fx::split(c.y, e);
      sc[g * T * NN + r] = make_int4(re.x, re.y, im.x, im.y);
    }
    __syncthreads();
    if (!l.in) continue;
    long long pA[SG], pB[SG], mA[SG], mB[SG], iA[SG], iB[SG];  // sums of a c, b d, (a + b)(c + d)
#pragma unroll
    for (int g = 0; g < SG; ++g) pA[g] = pB[g] = mA[g] = mB[g] = iA[g] = iB[g] = 0;
    const int4 *q = wq + slot * T * N, *c = sc + l.j;
#pragma unroll 1
    for (int t = 0; t < nb * N; ++t) {
      const int4 w = q[t];
      const int sx = w.x + w.z, sy = w.y + w.w;
#pragma unroll
      for (int g = 0; g < SG; ++g) {
        const int4 u = c[g * T * NN + t * N];
        fx::mac2(pA[g], pB[g], u.x, u.y, w.x, w.y);
        fx::mac2(mA[g], mB[g], u.z, u.w, w.z, w.w);
        fx::mac2(iA[g], iB[g], u.x + u.z, u.y + u.w, sx, sy);
      }
    }
#pragma unroll
    for (int g = 0; g < SG; ++g) {
      if (b >= nblk[g]) continue;
      const int e = ce[g * N + l.j], k = (ef - 1022) + (e - 1022) - 56;
      if (ef == 0x7ff || e == 0x7ff) {
        acc[g].x = acc[g].y = __longlong_as_double(0x7ff8000000000000LL);
      } else {
        const long long re = fx::join(pA[g] - mA[g], pB[g] - mB[g]);
        const long long im = fx::join(iA[g] - pA[g] - mA[g], iB[g] - pB[g] - mB[g]);
        bool small = ef && e && !fx::reaches(re, im, 56 - kFar);  // (largest times largest: 2^54 to 2^56)
        if (small) {
          unsigned size = 0;  // (largest times largest: 2^22 to 2^24)
#pragma unroll 1
          for (int t = 0; t < nb * N; ++t) {
            const int4 w = q[t], u = c[g * T * NN + t * N];
            size += (unsigned)((abs(w.x) + abs(w.z)) >> 16) * (unsigned)((abs(u.x) + abs(u.z)) >> 16);
          }
          small = size < 1u << (24 - kFar);
        }
        if (small) {
          const double2 z = basis64_terms<N>(basis, b, min(nb, nblk[g] - b), l.row, l.j,
                                             cf + ((size_t)(s0 - 1 + g) * cfstride + b) * NN);
          acc[g].x += z.x;
          acc[g].y += z.y;
        } else {
          acc[g].x += fx::value(re, k);
          acc[g].y += fx::value(im, k);
        }
      }
    }
  }
  if (!l.in) return;
#pragma unroll
  for (int g = 0; g < SG; ++g)
    if (s0 + g < nshift && (want != 1 || nblk[g])) out[(size_t)(s0 - 1 + g) * fstride + l.row * N + l.j] = acc[g];
}

rhmc_status_t axpy64(const double2 *A, double2 *const *basis, const int *kdev, const double2 *M, double2 *Y, long rows,
                     int n, cudaStream_t s) {
  prof_begin(PROF_AXPY, s);
#define L_(NN)                                                                                          \
  {                                                                                                     \
    const long grid = std::min<long>((rows + 4 * Lanes<NN>::RPW - 1) / (4 * Lanes<NN>::RPW), 16 * 152); \
    k_axpy64<NN><<<(unsigned)grid, 128, 0, s>>>(A, basis, kdev, M, Y, rows);                            \
  }
  RHMC_DISPATCH_N(n, L_)
#undef L_
  prof_end(s, (double)rows * n * sizeof(double2) * 3);
  RHMC_LAUNCH_CHECK();
  return RHMC_OK;
}

rhmc_status_t base64(const double2 *W, double2 *const *basis, const int *kdev, double2 *P, double2 *X, const double2 *coef,
                     long rows, int n, cudaStream_t s) {
  prof_begin(PROF_UPDATE64, s);
#define L_(NN)                                                                                          \
  {                                                                                                     \
    const long grid = std::min<long>((rows + 4 * Lanes<NN>::RPW - 1) / (4 * Lanes<NN>::RPW), 16 * 152); \
    k_base64<NN><<<(unsigned)grid, 128, 0, s>>>(W, basis, kdev, P, X, coef, rows);                      \
  }
  RHMC_DISPATCH_N(n, L_)
#undef L_
  prof_end(s, (double)rows * n * sizeof(double2) * 6);
  RHMC_LAUNCH_CHECK();
  return RHMC_OK;
}

template <int N, int SG>
static void launch_apply(const BasisBufs &bb, double2 *const *basis, const double2 *cf, int nshift,
                         const SolverState *st, long rows, int K, int want, double2 *out, long fstride,
                         cudaStream_t s) {
  const dim3 grid((unsigned)((rows + 4 * Lanes<N>::RPW - 1) / (4 * Lanes<N>::RPW)), (unsigned)((nshift - 2 + SG) / SG));
  k_basis64_apply<N, SG><<<grid, 128, 0, s>>>(basis, rows, st, K, want, nshift, cf, bb.cap + 1, out, fstride);
}

rhmc_status_t basis64_assemble(const BasisBufs &bb, double2 *const *basis, int n, int nshift, const SolverState *st,
                               long rows, int K, int want_p, int combine, double2 *out, long fstride, cudaStream_t s) {
  if (nshift < 2 || (K <= 0 && !want_p)) return RHMC_OK;
  RHMC_TRY(basis_coef(bb, n, nshift, st, K, want_p, s));
  const double2 *cf = bb.cf;
  int ns = nshift, want = want_p;
  if (combine && !want_p) {
    double2 *sum = bb.cf + (size_t)(nshift - 1) * (bb.cap + 1) * n * n;
    k_basis64_combine<<<K, 256, 0, s>>>(n, nshift, st, K, bb.cf, bb.cap + 1, sum);
    RHMC_LAUNCH_CHECK();
    cf = sum;
    ns = 2;
    want = 2;
  }
  prof_begin(PROF_UPDATE64, s);
#define L_(NN)                                                                                   \
  if (ns > 2)                                                                                    \
    launch_apply<NN, 4>(bb, basis, cf, ns, st, rows, K, want, out, fstride, s);                  \
  else                                                                                           \
    launch_apply<NN, 1>(bb, basis, cf, ns, st, rows, K, want, out, fstride, s)
  RHMC_DISPATCH_N(n, L_)
#undef L_
  prof_end(s, (double)rows * n * sizeof(double2) * (K + ns - 1.0));
  RHMC_LAUNCH_CHECK();
  return RHMC_OK;
}

}  // namespace rhmc
