// Multi-RHS even-odd staggered hop (Sec. IV operator; block "pencil"
// application of Sec. III / conclusions: each gauge link is loaded once for
// all n right-hand sides).
//
// Internal link layout, one array per output parity p:
//   L_p[h][d][3][3], h = rank of the output site x among parity p,
//   d = mu       : eta_mu(x) b_mu(x) U_mu(x)                (forward, x+mu)
//   d = 4 + mu   : -eta_mu(x) b_mu(x-mu) U_mu(x-mu)^dagger   (backward, x-mu)
// so that (D psi)(x) = sum_d L_p[h][d] psi(nb_d(x)).  The 72 complex numbers a
// site needs are contiguous: a CTA stages the records of its site tile into
// shared memory with coalesced 16-byte loads and every thread of the tile (one
// per (site, right-hand side)) reads them from there.
#include <cstring>
#include <mutex>

#include "common.cuh"
#include "df.cuh"
#include "fx.cuh"
#include "kernels.h"

namespace rhmc {

// ------------------------------------------------------------ link staging
template <typename T>
__global__ void k_stage_links(Geom g, int par, const double2 *__restrict__ U, int bc_t, C<T> *__restrict__ out) {
  const long h = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (h >= g.Vh) return;
  int x[4];
  site_coords(g, par, h, x);
  const long lex = lex_of(g, x);
  C<T> *o = out + h * 72;
  int sum = 0;
  for (int mu = 0; mu < 4; ++mu) {
    const double eta = (sum & 1) ? -1.0 : 1.0;
    sum += x[mu];
    // forward link U_mu(x)
    const double bf = (mu == 3 && bc_t == -1 && x[3] == g.L[3] - 1) ? -1.0 : 1.0;
    const double2 *u = U + (lex * 4 + mu) * 9;
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) {
        const double2 z = u[a * 3 + b];
        o[mu * 9 + a * 3 + b] = mk<T>((T)(eta * bf * z.x), (T)(eta * bf * z.y));
      }
    // backward link U_mu(x-mu)^dagger
    int y[4] = {x[0], x[1], x[2], x[3]};
    y[mu] = (x[mu] == 0) ? g.L[mu] - 1 : x[mu] - 1;
    const double bb = (mu == 3 && bc_t == -1 && y[3] == g.L[3] - 1) ? -1.0 : 1.0;
    const double2 *v = U + (lex_of(g, y) * 4 + mu) * 9;
    for (int a = 0; a < 3; ++a)
      for (int b = 0; b < 3; ++b) {
        const double2 z = v[b * 3 + a];  // dagger: transpose + conjugate
        o[(4 + mu) * 9 + a * 3 + b] = mk<T>((T)(-eta * bb * z.x), (T)(eta * bb * z.y));
      }
  }
}

rhmc_status_t stage_links(const Geom &g, const double2 *U, int bc_t, double2 *l64[2], float2 *l32[2],
                          cudaStream_t s) {
  const int bs = 128;
  const int grid = (int)((g.Vh + bs - 1) / bs);
  for (int p = 0; p < 2; ++p) {
    k_stage_links<double><<<grid, bs, 0, s>>>(g, p, U, bc_t, l64[p]);
    RHMC_LAUNCH_CHECK();
    k_stage_links<float><<<grid, bs, 0, s>>>(g, p, U, bc_t, l32[p]);
    RHMC_LAUNCH_CHECK();
  }
  return RHMC_OK;
}

// Coordinates of the site with parity `par` and parity rank h, 32-bit
// arithmetic (V/2 < 2^31): x = 2 xh + (parity of y + z + t xor par).
__device__ __forceinline__ void site_coords32(const Geom &g, int par, int h, int &x0, int &x1, int &x2, int &x3) {
  const int r = h / g.Lxh;
  const int xh = h - r * g.Lxh;
  const int r2 = r / g.L[1];
  x1 = r - r2 * g.L[1];
  x3 = r2 / g.L[2];
  x2 = r2 - x3 * g.L[2];
  x0 = 2 * xh + (((x1 + x2 + x3) & 1) ^ par);
}

// ------------------------------------------------------------ 12-real links
// A link record L = f V with V in SU(3) and f = +-1 (f = eta b for the forward
// links, f = -eta b for the daggered backward ones) is determined by its first
// two rows: row 3 = f conj(row 1 x row 2).  The FP32 hop can therefore read 6
// of the 9 complex entries (384 instead of 576 bytes per site) and rebuild the
// third rows in shared memory.  The sign of record d of the site with parity
// `par` and coordinates x:
__device__ __forceinline__ float link_sign(const Geom &g, int bc_t, int d, int x0, int x1, int x2, int x3) {
  const int mu = d & 3;
  const int ps = mu == 0 ? 0 : mu == 1 ? x0 : mu == 2 ? x0 + x1 : x0 + x1 + x2;
  float f = (ps & 1) ? -1.f : 1.f;  // eta_mu(x)
  if (d < 4) {
    if (mu == 3 && bc_t == -1 && x3 == g.L[3] - 1) f = -f;  // b_mu(x)
  } else {
    if (mu == 3 && bc_t == -1 && x3 == 0) f = -f;  // b_mu(x - mu)
    f = -f;
  }
  return f;
}

__device__ __forceinline__ float2 cross_conj(float2 a1, float2 a2, float2 b1, float2 b2) {
  // conj(a1 b2 - a2 b1)
  const float re = a1.x * b2.x - a1.y * b2.y - (a2.x * b1.x - a2.y * b1.y);
  const float im = a1.x * b2.y + a1.y * b2.x - (a2.x * b1.y + a2.y * b1.x);
  return make_float2(re, -im);
}

// first two rows of every FP32 record; *dev_max = largest |row 3 - rebuilt row 3|
__global__ void k_links12(Geom g, int par, int bc_t, const float2 *__restrict__ l32, float2 *__restrict__ l12,
                          unsigned *dev_max) {
  const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;  // (site, d)
  if (k >= g.Vh * 8) return;
  const int h = (int)(k >> 3), d = (int)(k & 7);
  const float2 *L = l32 + k * 9;
  float2 r[6];
#pragma unroll
  for (int e = 0; e < 6; ++e) {
    r[e] = L[e];
    l12[k * 6 + e] = r[e];
  }
  int x0, x1, x2, x3;
  site_coords32(g, par, h, x0, x1, x2, x3);
  const float f = link_sign(g, bc_t, d, x0, x1, x2, x3);
  float dev = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
    const float2 t = cross_conj(r[c1], r[c2], r[3 + c1], r[3 + c2]);
    const float2 w = L[6 + c];
    dev = fmaxf(dev, fmaxf(fabsf(w.x - f * t.x), fabsf(w.y - f * t.y)));
  }
  atomicMax(dev_max, __float_as_uint(dev));  // non-negative floats order as their bit patterns
}

// ------------------------------------------------------------ hop
// out[b] = D in[b]                 (self == nullptr)
// out[b] = a self[b] - D in[b]     (the fused 4m^2 + sigma axpy of A)
// on parity `par`, for nbatch independent fields b (stride bstride) that
// share the staged links.
//
// Thread layout: R right-hand sides per thread (register blocking), n / R
// threads per site, `tile` sites per CTA.  The CTA stages the 72-complex link
// records of its sites into shared memory once, together with the 8 neighbour
// offsets of each site.  The loop over the 8 directions keeps the next
// direction's neighbour block in flight while the current one is multiplied.
namespace {


template <typename T> __device__ __forceinline__ void lmac(C<T> &acc, const C<T> &e, const C<T> &v) {
  cmac<T>(acc, e, v);
}

template <typename T> struct LinkSlot { using t = C<T>; };

template <typename T> __device__ __forceinline__ void expand(C<T> &dst, C<T> z) { dst = z; }

// Vector load / store of R consecutive complex numbers.
template <typename T, int R> struct Vec;
template <> struct Vec<float, 4> {
  __device__ static void ld(const float2 *p, float2 *v) {
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p)), b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
    v[0] = make_float2(a.x, a.y); v[1] = make_float2(a.z, a.w); v[2] = make_float2(b.x, b.y); v[3] = make_float2(b.z, b.w);
  }
  __device__ static void st(float2 *p, const float2 *v) {
    reinterpret_cast<float4 *>(p)[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
    reinterpret_cast<float4 *>(p)[1] = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
  }
};
template <> struct Vec<float, 2> {
  __device__ static void ld(const float2 *p, float2 *v) {
    const float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    v[0] = make_float2(a.x, a.y); v[1] = make_float2(a.z, a.w);
  }
  __device__ static void st(float2 *p, const float2 *v) {
    reinterpret_cast<float4 *>(p)[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  }
};
template <typename T> struct Vec1 {
  __device__ static void ld(const C<T> *p, C<T> *v) { v[0] = p[0]; }
  __device__ static void st(C<T> *p, const C<T> *v) { p[0] = v[0]; }
};
template <> struct Vec<float, 1> : Vec1<float> {};
template <> struct Vec<double, 1> : Vec1<double> {};
template <int R> struct VecD {
  __device__ static void ld(const double2 *p, double2 *v) {
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = __ldg(p + r);
  }
  __device__ static void st(double2 *p, const double2 *v) {
#pragma unroll
    for (int r = 0; r < R; ++r) p[r] = v[r];
  }
};
template <> struct Vec<double, 2> : VecD<2> {};
template <> struct Vec<double, 4> : VecD<4> {};

}  // namespace

template <typename T, int R, bool SELF, bool STAGE>
__global__ void __launch_bounds__(128) k_hop(Geom g, int par, const C<T> *__restrict__ links,
                                             const C<T> *__restrict__ in, C<T> *__restrict__ out,
                                             const C<T> *__restrict__ self, T a, int n, int tile, int nbatch,
                                             long bstride) {
  using LS = typename LinkSlot<T>::t;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  LS *sl = reinterpret_cast<LS *>(smem_raw);
  const int tps = n / R;
  const int h0 = blockIdx.x * tile;
  const int nsites = min(tile, (int)g.Vh - h0);
  if (STAGE) {
    const C<T> *src = links + (long)h0 * 72;
    for (int k = threadIdx.x; k < nsites * 72; k += blockDim.x) expand<T>(sl[k], __ldg(src + k));
    __syncthreads();
  }
  // neighbour ranks of every site of the tile, shared by the site's threads
  int *snb = reinterpret_cast<int *>(smem_raw + (STAGE ? (size_t)tile * 72 * sizeof(LS) : 0));
  for (int k = threadIdx.x; k < nsites * 8; k += blockDim.x) {
    const int site = k >> 3, d = k & 7;
    int x[4];
    site_coords(g, par, h0 + site, x);
    const int mu = d & 3, st = d < 4 ? 1 : -1;
    // neighbour coordinates without dynamic indexing of x[]
    int y0 = x[0], y1 = x[1], y2 = x[2], y3 = x[3];
    if (mu == 0) y0 = (y0 + st + g.L[0]) % g.L[0];
    else if (mu == 1) y1 = (y1 + st + g.L[1]) % g.L[1];
    else if (mu == 2) y2 = (y2 + st + g.L[2]) % g.L[2];
    else y3 = (y3 + st + g.L[3]) % g.L[3];
    const int lex = y0 + g.L[0] * (y1 + g.L[1] * (y2 + g.L[2] * y3));
    snb[k] = (lex >> 1) * 3 * n;
  }
  __syncthreads();
  const int ls = threadIdx.x / tps;
  const int j0 = (threadIdx.x - ls * tps) * R;
  if (ls >= nsites) return;
  const int h = h0 + ls;
  const int o = h * 3 * n + j0;
  for (int b = 0; b < nbatch; ++b) {
    const C<T> *inb = in + b * bstride;
    C<T> acc[3][R];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int r = 0; r < R; ++r) acc[c][r] = czero<T>();
    C<T> v[3][R], vn[3][R];
#pragma unroll
    for (int c = 0; c < 3; ++c) Vec<T, R>::ld(inb + snb[ls * 8] + j0 + c * n, v[c]);
#pragma unroll 1
    for (int d = 0; d < 8; ++d) {
      // prefetch the next direction's neighbour block while this one is used
      const int dn = d < 7 ? d + 1 : d;
#pragma unroll
      for (int c = 0; c < 3; ++c) Vec<T, R>::ld(inb + snb[ls * 8 + dn] + j0 + c * n, vn[c]);
#pragma unroll
      for (int ca = 0; ca < 3; ++ca)
#pragma unroll
        for (int cb = 0; cb < 3; ++cb) {
          LS e;
          if (STAGE)
            e = sl[ls * 72 + d * 9 + ca * 3 + cb];
          else
            expand<T>(e, __ldg(links + (long)h * 72 + d * 9 + ca * 3 + cb));
#pragma unroll
          for (int r = 0; r < R; ++r) lmac<T>(acc[ca][r], e, v[cb][r]);
        }
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int r = 0; r < R; ++r) v[c][r] = vn[c][r];
    }
    C<T> *ob = out + b * bstride + o;
    if (SELF) {
      const C<T> *sb = self + b * bstride + o;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        C<T> sv[R];
        Vec<T, R>::ld(sb + c * n, sv);
#pragma unroll
        for (int r = 0; r < R; ++r) acc[c][r] = mk<T>(a * sv[r].x - acc[c][r].x, a * sv[r].y - acc[c][r].y);
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) Vec<T, R>::st(ob + c * n, acc[c]);
  }
}

template <typename T, int R>
static void launch_hop(const Geom &g, int par, const C<T> *links, const C<T> *in, C<T> *out, const C<T> *self,
                       double a, int n, int nbatch, long bstride, cudaStream_t s) {
  using LS = typename LinkSlot<T>::t;
  const int tps = n / R;
  const bool stage = tps >= 2;  // links are reused only when several threads share a site
  const int tile = max(1, 128 / tps);
  const int threads = ((tile * tps + 31) / 32) * 32;
  const size_t smem = (stage ? (size_t)tile * 72 * sizeof(LS) : 0) + (size_t)tile * 8 * sizeof(int);
  const unsigned grid = (unsigned)((g.Vh + tile - 1) / tile);
  static std::once_flag attr_done;
  std::call_once(attr_done, [&] {
    cudaFuncSetAttribute(k_hop<T, R, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    cudaFuncSetAttribute(k_hop<T, R, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    cudaFuncSetAttribute(k_hop<T, R, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    cudaFuncSetAttribute(k_hop<T, R, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
  });
  if (self) {
    if (stage)
      k_hop<T, R, true, true><<<grid, threads, smem, s>>>(g, par, links, in, out, self, (T)a, n, tile, nbatch, bstride);
    else
      k_hop<T, R, true, false><<<grid, threads, smem, s>>>(g, par, links, in, out, self, (T)a, n, tile, nbatch, bstride);
  } else {
    if (stage)
      k_hop<T, R, false, true><<<grid, threads, smem, s>>>(g, par, links, in, out, self, (T)a, n, tile, nbatch, bstride);
    else
      k_hop<T, R, false, false><<<grid, threads, smem, s>>>(g, par, links, in, out, self, (T)a, n, tile, nbatch, bstride);
  }
}

// ------------------------------------------------------------ hop, all directions in flight
// FP32, one right-hand side per thread, n threads per site, TS = 128 / n sites
// per CTA.  The CTA's link records go to shared memory by cp.async while the
// neighbour table is built; then every thread issues the loads of all 8
// neighbours' 3 colour components at once (24 independent 8-byte loads, about
// 200 bytes per thread in flight) before it multiplies anything, so the
// latency of the gathered reads is paid once per site instead of once per
// direction.
template <int N, int R, bool SELF, bool REC>
__global__ void __launch_bounds__(128) k_hop_pf(Geom g, int par, const float2 *__restrict__ links,
                                                const float2 *__restrict__ in, float2 *__restrict__ out,
                                                const float2 *__restrict__ self, float a, int bc_t,
                                                const SolverState *__restrict__ st) {
  const int done = st ? st->done : 0;                        // (tested once the loads below are on their way)
  constexpr int TPS = N / R;                                 // threads per site
  constexpr int TILE = (128 / TPS) < 32 ? (128 / TPS) : 32;  // sites per CTA (static shared memory <= 20 KB)
  constexpr int LR = REC ? 48 : 72;  // complex per site record as stored
  __shared__ __align__(16) float2 sl[TILE * 72];
  __shared__ __align__(16) float2 sl12[REC ? TILE * 48 : 1];
  __shared__ float sgn[REC ? TILE * 8 : 1];
  __shared__ int snb[TILE * 8];
  const int tid = threadIdx.x;
  const int h0 = blockIdx.x * TILE;
  const int nsites = min(TILE, (int)g.Vh - h0);
  {
    const unsigned base = (unsigned)__cvta_generic_to_shared(REC ? sl12 : sl);
    const char *src = reinterpret_cast<const char *>(links + (long)h0 * LR);
    for (int c = tid; c < nsites * (LR / 2); c += blockDim.x)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(base + 16u * c), "l"(src + 16L * c) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int k = tid; k < nsites * 8; k += blockDim.x) {
    const int site = k >> 3, d = k & 7;
    int y0, y1, y2, y3;
    site_coords32(g, par, h0 + site, y0, y1, y2, y3);
    if (REC) sgn[k] = link_sign(g, bc_t, d, y0, y1, y2, y3);
    const int mu = d & 3;
    const bool fwd = d < 4;
    if (mu == 0) y0 = fwd ? (y0 + 1 == g.L[0] ? 0 : y0 + 1) : (y0 == 0 ? g.L[0] - 1 : y0 - 1);
    else if (mu == 1) y1 = fwd ? (y1 + 1 == g.L[1] ? 0 : y1 + 1) : (y1 == 0 ? g.L[1] - 1 : y1 - 1);
    else if (mu == 2) y2 = fwd ? (y2 + 1 == g.L[2] ? 0 : y2 + 1) : (y2 == 0 ? g.L[2] - 1 : y2 - 1);
    else y3 = fwd ? (y3 + 1 == g.L[3] ? 0 : y3 + 1) : (y3 == 0 ? g.L[3] - 1 : y3 - 1);
    const int lex = y0 + g.L[0] * (y1 + g.L[1] * (y2 + g.L[2] * y3));
    snb[k] = (lex >> 1) * 3 * N;
  }
  const double a_st = (SELF && st) ? st->a0 : 0.0;
  __syncthreads();
  if (done) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    return;
  }
  const int ls = tid / TPS, j = (tid - (tid / TPS) * TPS) * R;
  const bool live = ls < nsites;
  float2 v[8][3][R];
  if (live) {
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      const float2 *nb = in + snb[ls * 8 + d] + j;
#pragma unroll
      for (int c = 0; c < 3; ++c) Vec<float, R>::ld(nb + c * N, v[d][c]);
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  if (REC) {  // full records from the first two rows: row 3 = f conj(row 1 x row 2)
    for (int e = tid; e < nsites * 8; e += blockDim.x) {
      const float2 *r = sl12 + e * 6;
      float2 *o = sl + (e >> 3) * 72 + (e & 7) * 9;
      const float f = sgn[e];
#pragma unroll
      for (int c = 0; c < 6; ++c) o[c] = r[c];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
        const float2 t = cross_conj(r[c1], r[c2], r[3 + c1], r[3 + c2]);
        o[6 + c] = make_float2(f * t.x, f * t.y);
      }
    }
    __syncthreads();
  }
  if (!live) return;
  float2 acc[3][R];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int r = 0; r < R; ++r) acc[c][r] = make_float2(0.f, 0.f);
  const float2 *lk = sl + ls * 72;
#pragma unroll
  for (int d = 0; d < 8; ++d)
#pragma unroll
    for (int ca = 0; ca < 3; ++ca)
#pragma unroll
      for (int cb = 0; cb < 3; ++cb) {
        const float2 e = lk[d * 9 + ca * 3 + cb];
#pragma unroll
        for (int r = 0; r < R; ++r) cmac<float>(acc[ca][r], e, v[d][cb][r]);
      }
  float2 *op = out + (long)(h0 + ls) * 3 * N + j;
  if (SELF) {
    if (st) a = (float)a_st;
    const float2 *sp = self + (long)(h0 + ls) * 3 * N + j;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float2 sv[R];
      Vec<float, R>::ld(sp + c * N, sv);
#pragma unroll
      for (int r = 0; r < R; ++r) acc[c][r] = make_float2(a * sv[r].x - acc[c][r].x, a * sv[r].y - acc[c][r].y);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) Vec<float, R>::st(op + c * N, acc[c]);
}

template <int N, int R>
static void launch_hop_pf_n(const Geom &g, int par, const float2 *links, const float2 *in, float2 *out,
                            const float2 *self, double a, const float2 *links12, int bc_t, const SolverState *st,
                            cudaStream_t s) {
  constexpr int TPS = N / R;
  constexpr int TILE = (128 / TPS) < 32 ? (128 / TPS) : 32;
  const int threads = ((TILE * TPS + 31) / 32) * 32;
  const unsigned grid = (unsigned)((g.Vh + TILE - 1) / TILE);
  if (links12) {
    if (self)
      k_hop_pf<N, R, true, true><<<grid, threads, 0, s>>>(g, par, links12, in, out, self, (float)a, bc_t, st);
    else
      k_hop_pf<N, R, false, true><<<grid, threads, 0, s>>>(g, par, links12, in, out, self, (float)a, bc_t, st);
  } else if (self) {
    k_hop_pf<N, R, true, false><<<grid, threads, 0, s>>>(g, par, links, in, out, self, (float)a, bc_t, st);
  } else {
    k_hop_pf<N, R, false, false><<<grid, threads, 0, s>>>(g, par, links, in, out, self, (float)a, bc_t, st);
  }
}

static bool launch_hop_pf(const Geom &g, int par, const float2 *links, const float2 *in, float2 *out,
                          const float2 *self, double a, int n, const float2 *links12, int bc_t,
                          const SolverState *st, cudaStream_t s) {
  // two right-hand sides per thread (16-byte loads, half the load instructions): built-in
  // for even n >= 12 (measured at 24^4: n = 16 65 us against 71 us; n = 8 no gain)
  const int mode = tune_get(TUNE_HOP_STAGED);
  const bool r2 = n % 2 == 0 && (mode == 4 || (mode == 0 && n >= 12));
  switch (n) {
#define L_PF(NN)                                                                   \
  case NN:                                                                         \
    if constexpr (NN % 2 == 0) {                                                   \
      if (r2) {                                                                    \
        launch_hop_pf_n<NN, 2>(g, par, links, in, out, self, a, links12, bc_t, st, s); \
        return true;                                                               \
      }                                                                            \
    }                                                                              \
    launch_hop_pf_n<NN, 1>(g, par, links, in, out, self, a, links12, bc_t, st, s);     \
    return true;
    L_PF(1) L_PF(2) L_PF(3) L_PF(4) L_PF(5) L_PF(6) L_PF(7) L_PF(8)
    L_PF(9) L_PF(10) L_PF(11) L_PF(12) L_PF(13) L_PF(14) L_PF(15) L_PF(16)
#undef L_PF
    default: return false;
  }
}

// ------------------------------------------------------------ hop, cp.async staged
// FP32, one field, even n: persistent CTAs walk over tiles of TS output sites.
// All threads stage the next tile into shared memory with 16-byte cp.async
// copies (L2 only) while the current tile is multiplied:
//   the TS link records (TS * 72 complex, contiguous),
//   the 8 neighbour rows of every site (3n complex each, gathered),
//   the TS rows of `self` for the fused axpy (contiguous).
// Two buffers, one cp.async group per tile, so every thread keeps a whole
// tile's share of loads in flight without holding them in registers.  Every
// thread owns R right-hand sides of one site.
namespace {
template <int R> struct SVec;  // shared-memory vector loads
template <> struct SVec<1> {
  __device__ static void ld(const float2 *p, float2 *v) { v[0] = p[0]; }
};
template <> struct SVec<2> {
  __device__ static void ld(const float2 *p, float2 *v) {
    const float4 a = *reinterpret_cast<const float4 *>(p);
    v[0] = make_float2(a.x, a.y);
    v[1] = make_float2(a.z, a.w);
  }
};
template <> struct SVec<4> {
  __device__ static void ld(const float2 *p, float2 *v) {
    SVec<2>::ld(p, v);
    SVec<2>::ld(p + 2, v + 2);
  }
};
__device__ __forceinline__ void cp_async16(unsigned dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
}  // namespace

template <int R, bool SELF>
__global__ void __launch_bounds__(128) k_hop_staged(Geom g, int par, const float2 *__restrict__ links,
                                                    const float2 *__restrict__ in, float2 *__restrict__ out,
                                                    const float2 *__restrict__ self, float a, int n, int TS,
                                                    int ntiles) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int tps = n / R;
  const int row = 3 * n;      // complex numbers of one site row
  const int cpr = 3 * n / 2;  // 16-byte chunks of one site row
  const unsigned link_b = (unsigned)TS * 72 * 8, nb_b = (unsigned)TS * 8 * row * 8;
  const unsigned stage_b = link_b + nb_b + (SELF ? (unsigned)TS * row * 8 : 0u);
  int *snb = reinterpret_cast<int *>(smem_raw + 2 * stage_b);  // [2][TS * 8] neighbour ranks
  const int nthr = blockDim.x, tid = threadIdx.x;
  // per-thread walk over (row, chunk) pairs: start and stride without divisions in the loop
  const int q0 = tid % cpr, r0 = tid / cpr, dq = nthr % cpr, dr = nthr / cpr;

  auto fill_nb = [&](int tile, int buf) {
    const int h0 = tile * TS;
    const int ns = min(TS, (int)g.Vh - h0);
    for (int k = tid; k < ns * 8; k += nthr) {
      const int site = k >> 3, d = k & 7;
      int x[4];
      site_coords(g, par, h0 + site, x);
      const int mu = d & 3, st = d < 4 ? 1 : -1;
      int y0 = x[0], y1 = x[1], y2 = x[2], y3 = x[3];
      if (mu == 0) y0 = (y0 + st + g.L[0]) % g.L[0];
      else if (mu == 1) y1 = (y1 + st + g.L[1]) % g.L[1];
      else if (mu == 2) y2 = (y2 + st + g.L[2]) % g.L[2];
      else y3 = (y3 + st + g.L[3]) % g.L[3];
      const int lex = y0 + g.L[0] * (y1 + g.L[1] * (y2 + g.L[2] * y3));
      snb[buf * TS * 8 + k] = lex >> 1;
    }
  };
  auto issue = [&](int tile, int buf) {
    const int h0 = tile * TS;
    const int ns = min(TS, (int)g.Vh - h0);
    const unsigned base = (unsigned)__cvta_generic_to_shared(smem_raw + buf * stage_b);
    const char *lsrc = reinterpret_cast<const char *>(links + (long)h0 * 72);
    for (int c = tid; c < ns * 36; c += nthr) cp_async16(base + 16u * c, lsrc + 16L * c);
    const int *nb = snb + buf * TS * 8;
    int q = q0, r = r0;
    while (r < ns * 8) {
      cp_async16(base + link_b + (unsigned)(r * row * 8 + q * 16),
                 reinterpret_cast<const char *>(in + (long)nb[r] * row) + 16 * q);
      q += dq;
      r += dr;
      if (q >= cpr) {
        q -= cpr;
        ++r;
      }
    }
    if (SELF) {
      const char *ssrc = reinterpret_cast<const char *>(self + (long)h0 * row);
      for (int c = tid; c < ns * cpr; c += nthr) cp_async16(base + link_b + nb_b + 16u * c, ssrc + 16L * c);
    }
  };
  const int ls = tid / tps;
  const int j0 = (tid - ls * tps) * R;
  int tile = blockIdx.x;
  if (tile < ntiles) {
    fill_nb(tile, 0);
    __syncthreads();
    issue(tile, 0);
  }
  cp_async_commit();
  for (int i = 0; tile < ntiles; tile += gridDim.x, ++i) {
    const int buf = i & 1;
    const int next = tile + gridDim.x;
    if (next < ntiles) fill_nb(next, buf ^ 1);
    __syncthreads();  // neighbour table ready; buffer buf ^ 1 no longer read
    if (next < ntiles) issue(next, buf ^ 1);
    cp_async_commit();
    cp_async_wait<1>();  // this thread's copies of the current tile landed
    __syncthreads();     // ... and everyone else's
    const int h0 = tile * TS;
    const int ns = min(TS, (int)g.Vh - h0);
    if (ls < ns) {
      const unsigned char *sb = smem_raw + buf * stage_b;
      const float2 *sl = reinterpret_cast<const float2 *>(sb) + ls * 72;
      const float2 *sn = reinterpret_cast<const float2 *>(sb + link_b) + ls * 8 * row + j0;
      float2 acc[3][R];
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int r = 0; r < R; ++r) acc[c][r] = make_float2(0.f, 0.f);
#pragma unroll 2
      for (int d = 0; d < 8; ++d) {
        float2 v[3][R];
#pragma unroll
        for (int c = 0; c < 3; ++c) SVec<R>::ld(sn + d * row + c * n, v[c]);
#pragma unroll
        for (int ca = 0; ca < 3; ++ca)
#pragma unroll
          for (int cb = 0; cb < 3; ++cb) {
            const float2 e = sl[d * 9 + ca * 3 + cb];
#pragma unroll
            for (int r = 0; r < R; ++r) cmac<float>(acc[ca][r], e, v[cb][r]);
          }
      }
      const long o = (long)(h0 + ls) * row + j0;
      if (SELF) {
        const float2 *ss = reinterpret_cast<const float2 *>(sb + link_b + nb_b) + ls * row + j0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          float2 sv[R];
          SVec<R>::ld(ss + c * n, sv);
#pragma unroll
          for (int r = 0; r < R; ++r) acc[c][r] = make_float2(a * sv[r].x - acc[c][r].x, a * sv[r].y - acc[c][r].y);
        }
      }
#pragma unroll
      for (int c = 0; c < 3; ++c) Vec<float, R>::st(out + o + c * n, acc[c]);
    }
  }
  cp_async_wait<0>();
}

template <int R>
static bool launch_hop_staged(const Geom &g, int par, const float2 *links, const float2 *in, float2 *out,
                              const float2 *self, double a, int n, cudaStream_t s) {
  const int tps = n / R;
  const long per_site = 576 + 8L * 24 * n + (self ? 24L * n : 0);
  const int TS = (int)std::min<long>(128 / tps, (96 * 1024) / per_site);
  if (TS < 1) return false;
  const int threads = ((TS * tps + 31) / 32) * 32;
  const size_t smem = 2 * (size_t)TS * per_site + 2 * (size_t)TS * 8 * sizeof(int);
  const int ntiles = (int)((g.Vh + TS - 1) / TS);
  static std::once_flag attr_done;
  std::call_once(attr_done, [] {
    cudaFuncSetAttribute(k_hop_staged<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 210 * 1024);
    cudaFuncSetAttribute(k_hop_staged<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 210 * 1024);
  });
  const int resident = self ? resident_ctas(k_hop_staged<R, true>, threads, smem)
                            : resident_ctas(k_hop_staged<R, false>, threads, smem);
  const int grid = std::min(ntiles, resident);
  if (self)
    k_hop_staged<R, true><<<grid, threads, smem, s>>>(g, par, links, in, out, self, (float)a, n, TS, ntiles);
  else
    k_hop_staged<R, false><<<grid, threads, smem, s>>>(g, par, links, in, out, self, (float)a, n, TS, ntiles);
  return true;
}

// The all-directions-in-flight kernel: FP32 single fields, the built-in choice
// (RHMC_TUNE_HOP_STAGED 0 or 3; 2 selects the register-staged kernel).
template <typename T> static bool use_hop_pf(const void *links, const void *in, int nbatch) {
  if (sizeof(C<T>) != 8 || nbatch != 1 || ((uintptr_t)links & 15)) return false;
  const int mode = tune_get(TUNE_HOP_STAGED);
  return mode == 0 || mode == 3 || mode == 4;  // 3: one right-hand side per thread, 4: two
}

// The staged kernel applies to FP32 single fields with 16-byte aligned rows.
template <typename T>
static bool try_hop_staged(const Geom &g, int par, const C<T> *links, const C<T> *in, C<T> *out,
                           const C<T> *self, double a, int n, int nbatch, int R, cudaStream_t s) {
  if constexpr (sizeof(C<T>) != 8) {
    return false;
  } else {
    const int mode = tune_get(TUNE_HOP_STAGED);
    // built-in: the register-staged kernel (measured faster at 24^4, n = 8 and 16)
    if (mode != 1 || nbatch != 1 || n % 2) return false;
    auto al16 = [](const void *p) { return ((uintptr_t)p & 15) == 0; };
    if (!al16(links) || !al16(in) || !al16(out) || (self && !al16(self))) return false;
    const float2 *L = reinterpret_cast<const float2 *>(links), *X = reinterpret_cast<const float2 *>(in),
                 *S = reinterpret_cast<const float2 *>(self);
    float2 *Y = reinterpret_cast<float2 *>(out);
    if (R == 4) return launch_hop_staged<4>(g, par, L, X, Y, S, a, n, s);
    if (R == 2) return launch_hop_staged<2>(g, par, L, X, Y, S, a, n, s);
    return launch_hop_staged<1>(g, par, L, X, Y, S, a, n, s);
  }
}

template <typename T>
rhmc_status_t hop(const Geom &g, int par, const C<T> *links, const C<T> *in, C<T> *out, const C<T> *self, double a,
                  int n, int nbatch, long bstride, cudaStream_t s, const C<T> *links12, int bc_t,
                  const SolverState *st) {
  if (n < 1 || n > RHMC_MAX_NRHS || g.Vh * 3L * n > 0x7fffffffL) return RHMC_ERR_INVALID_ARG;
  prof_begin(sizeof(T) == 4 ? PROF_HOP32 : PROF_HOP64, s);
  int R = tune_get(TUNE_HOP_RHS_PER_THREAD);
  // measured at 24^4 (FP32): 2 per thread best for n >= 12, 1 otherwise; FP64 is ALU bound
  if (R <= 0 || n % R != 0) R = (sizeof(T) == 4 && n >= 12 && n % 2 == 0) ? 2 : 1;
  if (try_hop_staged<T>(g, par, links, in, out, self, a, n, nbatch, R, s)) {
  } else if (use_hop_pf<T>(links, in, nbatch)) {
    launch_hop_pf(g, par, reinterpret_cast<const float2 *>(links), reinterpret_cast<const float2 *>(in),
                  reinterpret_cast<float2 *>(out), reinterpret_cast<const float2 *>(self), a, n,
                  reinterpret_cast<const float2 *>(links12), bc_t, st, s);
  } else if (R == 4)
    launch_hop<T, 4>(g, par, links, in, out, self, a, n, nbatch, bstride, s);
  else if (R == 2)
    launch_hop<T, 2>(g, par, links, in, out, self, a, n, nbatch, bstride, s);
  else
    launch_hop<T, 1>(g, par, links, in, out, self, a, n, nbatch, bstride, s);
  // algorithmic bytes: every link once, every input field once, the output once (+ self)
  prof_end(s, (double)g.Vh * sizeof(C<T>) * (72.0 + nbatch * 3.0 * n * (self ? 3 : 2)));
  RHMC_LAUNCH_CHECK();
  return RHMC_OK;
}

using namespace df;

// ------------------------------------------------------------ FP64-accurate hop on the integer units
// The FP64 operator, the residuals of the solvers and the force's D_oe X: sums of
// 24 complex products per output, formed exactly as integers (fx.cuh).  A field is
// converted once (k_fx_convert; the first hop of an operator application writes its
// result in integer form already), not by each of the eight neighbours that read it:
// converting inside the hop took 465 us per hop at 24^4, n = 16.
//
// Integer link records, one int4 per complex of the FP64 records, and the exponent of each
// site's largest entry (kSpecial where the site takes FP64 arithmetic: non-finite or zero
// links, or a row of one of them more than 2^3 below it, which never happens for SU(3)).
// Eight lanes per site, one per direction.
__global__ void __launch_bounds__(256) k_stage_links_fx(const double2 *__restrict__ l64, int4 *__restrict__ lfx,
                                                        int *__restrict__ lexp, long nrec) {
  const long k = (long)blockIdx.x * blockDim.x + threadIdx.x;  // (site, direction)
  const bool in = k < nrec;
  double2 v[9];
  int ef = 0, row = 0x7ff;  // largest exponent field; that of the smallest row
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    int er = 0;
#pragma unroll
    for (int e = 3 * a; e < 3 * a + 3; ++e) {
      v[e] = in ? l64[k * 9 + e] : make_double2(0.0, 0.0);
      er = max(er, max(fx::expo(v[e].x), fx::expo(v[e].y)));
    }
    ef = max(ef, er);
    row = min(row, er);
  }
#pragma unroll
  for (int off = 4; off > 0; off >>= 1) {
    ef = max(ef, __shfl_xor_sync(0xffffffffu, ef, off, 8));
    row = min(row, __shfl_xor_sync(0xffffffffu, row, off, 8));
  }
  if (!in) return;
#pragma unroll
  for (int e = 0; e < 9; ++e) {
    const int2 re = fx::split(v[e].x, ef), im = fx::split(v[e].y, ef);
    lfx[k * 9 + e] = make_int4(re.x, re.y, im.x, im.y);
  }
  if ((k & 7) == 0) lexp[k >> 3] = (ef == 0 || ef == 0x7ff || row < ef - 3) ? fx::kSpecial : ef - 1022;
}

rhmc_status_t stage_links_fx(const Geom &g, const double2 *l64, int4 *lfx, int *lexp, cudaStream_t s) {
  const long n = g.Vh * 8;
  k_stage_links_fx<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(l64, lfx, lexp, n);
  RHMC_LAUNCH_CHECK();
  return RHMC_OK;
}

// FP64 field [sites][3][n] -> integer form; one thread per (site, column)
__global__ void __launch_bounds__(128) k_fx_convert(const double2 *__restrict__ in, int4 *__restrict__ out,
                                                    int *__restrict__ ex, int count, int n) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  const int h = k / n;
  const long o = (long)h * 3 * n + (k - h * n);
  double2 v[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) v[c] = in[o + c * n];
  int4 q[3];
  ex[k] = fx::pack3(v, q);
#pragma unroll
  for (int c = 0; c < 3; ++c) out[o + c * n] = q[c];
}

static rhmc_status_t fx_convert(const Geom &g, const double2 *in, FxField out, int n, cudaStream_t s) {
  if (n < 1 || n > RHMC_MAX_NRHS || g.Vh * 3L * n > 0x7fffffffL) return RHMC_ERR_INVALID_ARG;
  const int count = (int)(g.Vh * n);
  prof_begin(PROF_OTHER, s);
  k_fx_convert<<<(unsigned)((count + 127) / 128), 128, 0, s>>>(in, out.v, out.e, count, n);
  prof_end(s, (double)count * (3 * 32.0 + 4.0));
  RHMC_LAUNCH_CHECK();
  return RHMC_OK;
}

// S lanes of a warp per (site, right-hand side), 8 / S directions each, `tile` sites per
// CTA.  The tile's link records go to shared memory by cp.async (padded to 73 int4,
// so that the sites of a warp read different banks).  A lane shifts each neighbour's
// words to the largest of the eight exponents and adds up its products: 648 integer
// multiply-adds of four clocks per (site, right-hand side), which bound the kernel
// on large lattices, and about 60 shifts and adds per direction on the other pipes.
// (Shifting every direction's sums instead took 350 us per hop at 24^4, n = 16,
// and 380 us without the three-product form.)  The loop over the directions
// is not unrolled: the unrolled body waited for the instruction cache.
// S = 4 where one lane per (site, right-hand side) would leave the schedulers without
// warps (small lattices): the lanes' integer sums are added by shuffles, and three of
// the four lanes write one colour each.  With S = 4 an FP64 input (IN64) is converted here:
// a separate pass would cost a launch, and each value is read by few warps.
// Measured, FP64 fields: 24^4, n = 16 787 us per operator application (60 us of it to convert
// the input of the first hop) against 2500 us with FP64 FMAs; at 8^4, n = 4 16 against 37 us.
// Against a long-double sum its error is 1.0e-16 relative for Gaussian fields, that of FP64 FMAs
// 2.9e-16.
// Lanes with a special block among their inputs, neighbours more than 2^26 apart in
// size, or an output whose terms are all small (fx.cuh) take FP64 arithmetic, on in64 where
// the input was given in FP64; its result is kept in FP64 (MODE 4).  In solves at 12^4, n = 4 the
// two hops take 11.5 and 13.2 us with the tests for that, 11.3 and 12.9 without; an input of one
// colour only (a source) 1.9 ms per operator application at 24^4, n = 16, and 2.6 ms under unit links.
//
// MODE 0: out = D in.  1: out = a self - D in.  2: out = B - (a self - D in), with
// the optional FP32 rounding outf and per-CTA column sums of |out|^2 (part).
// 3: out = D in as double-float pairs (float4).  4: D in in integer form, block words oex.
template <int MODE, int S, bool IN64>
__global__ void __launch_bounds__(128, 4) k_hop_fx(Geom g, int par, const int4 *__restrict__ lfx,
                                                   const int *__restrict__ lexp, const double2 *__restrict__ l64,
                                                   const int4 *__restrict__ in, const int *__restrict__ iex,
                                                   const double2 *__restrict__ in64, void *outv,
                                                   int *__restrict__ oex, const double2 *self, double a, int n,
                                                   int tile, const double2 *__restrict__ B, float2 *__restrict__ outf,
                                                   double *__restrict__ part) {
  constexpr int LS = 73;
  constexpr int IW = 32 / S;  // (site, right-hand side) items per warp
  constexpr int ND = 8 / S;   // directions per lane
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, nt = blockDim.x;
  int4 *sl = reinterpret_cast<int4 *>(smem_raw);
  int *snb = reinterpret_cast<int *>(sl + tile * LS);
  const int h0 = blockIdx.x * tile;
  const int nsites = min(tile, (int)g.Vh - h0);
  {
    const unsigned base = (unsigned)__cvta_generic_to_shared(sl);
    const char *src = reinterpret_cast<const char *>(lfx + (long)h0 * 72);
    for (int c = tid; c < nsites * 72; c += nt) {
      const int site = c / 72;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(base + 16u * (unsigned)(c + site)),
                   "l"(src + 16L * c)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int k = tid; k < nsites * 8; k += nt) {
    const int site = k >> 3, d = k & 7;
    int y0, y1, y2, y3;
    site_coords32(g, par, h0 + site, y0, y1, y2, y3);
    const int mu = d & 3;
    const bool fwd = d < 4;
    if (mu == 0) y0 = fwd ? (y0 + 1 == g.L[0] ? 0 : y0 + 1) : (y0 == 0 ? g.L[0] - 1 : y0 - 1);
    else if (mu == 1) y1 = fwd ? (y1 + 1 == g.L[1] ? 0 : y1 + 1) : (y1 == 0 ? g.L[1] - 1 : y1 - 1);
    else if (mu == 2) y2 = fwd ? (y2 + 1 == g.L[2] ? 0 : y2 + 1) : (y2 == 0 ? g.L[2] - 1 : y2 - 1);
    else y3 = fwd ? (y3 + 1 == g.L[3] ? 0 : y3 + 1) : (y3 == 0 ? g.L[3] - 1 : y3 - 1);
    const int lex = y0 + g.L[0] * (y1 + g.L[1] * (y2 + g.L[2] * y3));
    snb[k] = lex >> 1;
  }
  __syncthreads();
  const int lane = tid & 31, quad = lane / IW;  // which 8 / S of the directions
  const int item = (tid >> 5) * IW + (lane - quad * IW);
  const int ls = item / n, j = item - ls * n;
  const bool live = ls < nsites;
  const int *nb = snb + (live ? ls : 0) * 8;
  const int n3 = 3 * n, d0 = quad * ND;
  int E = fx::kZero, low = fx::kSpecial, even = fx::kZero, el = 0, ef = 0;  // even: the best neighbour's least colour
  int4 v[3];
  double2 x64[IN64 ? ND : 1][3];
  if (IN64) {
    bool any = false;
    if (live) {
      el = lexp[h0 + ls];
#pragma unroll
      for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int c = 0; c < 3; ++c) x64[IN64 ? d : 0][c] = __ldg(in64 + (nb[d0 + d] * n3 + j) + c * n);
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        int eb = 0, em = 0x7ff;
        bool some = false;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const double2 x = x64[IN64 ? d : 0][c];
          const int e = max(fx::expo(x.x), fx::expo(x.y));
          eb = max(eb, e);
          em = min(em, e);
          some = some || fx::nonzero(x.x) || fx::nonzero(x.y);
        }
        ef = max(ef, eb);
        if (em) even = max(even, em - 1022);
        if (some) low = min(low, eb - 1022);
        any = any || some;
      }
    }
#pragma unroll
    for (int off = IW; off < 32; off <<= 1) {
      ef = max(ef, __shfl_xor_sync(0xffffffffu, ef, off));
      any = __shfl_xor_sync(0xffffffffu, (int)any, off) || any;
    }
    E = !any ? fx::kZero : (ef == 0 || ef == 0x7ff) ? fx::kSpecial : ef - 1022;
  } else if (live) {
    el = lexp[h0 + ls];
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      const int code = iex[nb[d0 + d] * n + j], e = fx::exponent(code);
      E = max(E, e);
      low = min(low, e == fx::kZero ? fx::kSpecial : e);
      even = max(even, fx::least(code));
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) v[c] = __ldg(in + (nb[d0] * n3 + j) + c * n);
  }
#pragma unroll
  for (int off = IW; off < 32; off <<= 1) {
    if (!IN64) E = max(E, __shfl_xor_sync(0xffffffffu, E, off));
    low = min(low, __shfl_xor_sync(0xffffffffu, low, off));
    even = max(even, __shfl_xor_sync(0xffffffffu, even, off));
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  bool fast = E != fx::kSpecial && el != fx::kSpecial && (E == fx::kZero || E - low <= fx::kAlign);
  // colours apart at every neighbour: the sizes |U_cb| |v_b| themselves have to add up (fx.cuh)
  const bool unsure = live && fast && E != fx::kZero && E - even > fx::kApart;
  if (__any_sync(0xffffffffu, unsure)) {
    unsigned size[3] = {0, 0, 0};  // (units of 2^-24 of largest link times largest value)
    if (unsure) {
      const int4 *lk = sl + ls * LS + d0 * 9;
#pragma unroll 1
      for (int q = 0; q < 3 * ND; ++q) {
        const int d = q / 3, cb = q - d * 3, o = nb[d0 + d] * n3 + j + cb * n;
        int re, im;
        if (IN64) {
          re = fx::split(in64[o].x, ef).x;
          im = fx::split(in64[o].y, ef).x;
        } else {
          const int4 w = in[o];
          const int sh = min(fx::kAlign, E - fx::exponent(iex[nb[d0 + d] * n + j]));
          re = w.x >> sh;
          im = w.z >> sh;
        }
        const unsigned w = (unsigned)(abs(re) + abs(im)) >> 16;
#pragma unroll
        for (int ca = 0; ca < 3; ++ca) {
          const int4 l = lk[d * 9 + ca * 3 + cb];
          size[ca] += w * ((unsigned)(abs(l.x) + abs(l.z)) >> 16);
        }
      }
    }
#pragma unroll
    for (int off = IW; off < 32; off <<= 1)
#pragma unroll
      for (int c = 0; c < 3; ++c) size[c] += __shfl_xor_sync(0xffffffffu, size[c], off);
    if (unsure) fast = min(size[0], min(size[1], size[2])) >= 1u << 23;
  }
  long long R[6];
  if (live && fast) {
    long long pA[3], pB[3], mA[3], mB[3], iA[3], iB[3];  // sums of a c, b d, (a + b)(c + d)
#pragma unroll
    for (int c = 0; c < 3; ++c) pA[c] = pB[c] = mA[c] = mB[c] = iA[c] = iB[c] = 0;
    const int4 *lk = sl + ls * LS + d0 * 9;
    auto add = [&](int4 w, const int4 *l3) {  // one neighbour colour times the links' column
      const int sx = w.x + w.z, sy = w.y + w.w;
#pragma unroll
      for (int ca = 0; ca < 3; ++ca) {
        const int4 l = l3[ca * 3];
        fx::mac2(pA[ca], pB[ca], l.x, l.y, w.x, w.y);
        fx::mac2(mA[ca], mB[ca], l.z, l.w, w.z, w.w);
        fx::mac2(iA[ca], iB[ca], l.x + l.z, l.y + l.w, sx, sy);
      }
    };
    if constexpr (IN64) {
#pragma unroll
      for (int d = 0; d < ND; ++d)
#pragma unroll
        for (int cb = 0; cb < 3; ++cb) {
          const int2 re = fx::split(x64[d][cb].x, ef), im = fx::split(x64[d][cb].y, ef);
          add(make_int4(re.x, re.y, im.x, im.y), lk + d * 9 + cb);
        }
    } else {
#pragma unroll 1
      for (int d = d0; d < d0 + ND; ++d, lk += 9) {
        const int sh = min(fx::kAlign, E - fx::exponent(iex[nb[d] * n + j]));  // (clamped for zeros only)
        int4 w[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) w[c] = v[c];
        if (d < d0 + ND - 1) {  // the next direction's values are in flight while this one's are multiplied
          const int4 *p = in + (nb[d + 1] * n3 + j);
#pragma unroll
          for (int c = 0; c < 3; ++c) v[c] = __ldg(p + c * n);
        }
#pragma unroll
        for (int cb = 0; cb < 3; ++cb) {
          fx::align(w[cb].x, w[cb].y, sh);
          fx::align(w[cb].z, w[cb].w, sh);
          add(w[cb], lk + cb);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      R[2 * c] = fx::join(pA[c] - mA[c], pB[c] - mB[c]);
      R[2 * c + 1] = fx::join(iA[c] - pA[c] - mA[c], iB[c] - pB[c] - mB[c]);
    }
  } else {
#pragma unroll
    for (int c = 0; c < 6; ++c) R[c] = 0;
  }
#pragma unroll
  for (int off = IW; off < 32; off <<= 1)
#pragma unroll
    for (int c = 0; c < 6; ++c) R[c] += __shfl_xor_sync(0xffffffffu, R[c], off);
  double nrm = 0.0;
  if (live) {
    const int c0 = S == 1 ? 0 : quad, c1 = S == 1 ? 3 : min(3, quad + 1);  // this lane's colours
    const long o = (long)(h0 + ls) * n3 + j;
    const int k = E + el - 56;
    double2 acc[3];
    if (!fast) {
#pragma unroll
      for (int c = 0; c < 3; ++c) acc[c] = make_double2(0.0, 0.0);
      const double2 *L = l64 + (long)(h0 + ls) * 72;
#pragma unroll 1
      for (int q = 0; q < 24; ++q) {
        const int d = q / 3, cb = q - d * 3;
        const double2 w = IN64 || in64 ? in64[nb[d] * n3 + j + cb * n]
                                       : fx::unpack(in[nb[d] * n3 + j + cb * n], fx::exponent(iex[nb[d] * n + j]));
        const double2 *l = L + d * 9 + cb;
#pragma unroll
        for (int ca = 0; ca < 3; ++ca) cmac<double>(acc[ca], l[ca * 3], w);
      }
    }
    if (MODE == 4) {
      int4 q[3];
      int e;
      if (!fast) {
        e = fx::keep3(acc, q);
      } else if (E == fx::kZero) {
        e = fx::code(fx::kZero, 0);
        q[0] = q[1] = q[2] = make_int4(0, 0, 0, 0);
      } else {
        e = fx::renorm3(R, k, q);
      }
      if (quad == 0) oex[(long)(h0 + ls) * n + j] = e;
#pragma unroll
      for (int c = 0; c < 3; ++c)
        if (c >= c0 && c < c1) reinterpret_cast<int4 *>(outv)[o + c * n] = q[c];
      return;
    }
    double2 *out = reinterpret_cast<double2 *>(outv);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (c < c0 || c >= c1) continue;
      double2 r = fast ? make_double2(fx::value(R[2 * c], k), fx::value(R[2 * c + 1], k)) : acc[c];
      if (MODE == 1 || MODE == 2) {
        const double2 s = self[o + c * n];
        r = make_double2(fma(a, s.x, -r.x), fma(a, s.y, -r.y));
      }
      if (MODE == 2) {
        const double2 b = B[o + c * n];
        r = make_double2(b.x - r.x, b.y - r.y);
        if (outf) outf[o + c * n] = make_float2((float)r.x, (float)r.y);
        if (part) nrm = fma(r.x, r.x, fma(r.y, r.y, nrm));
      }
      if (MODE == 3) {
        const float2 x = df_split1(r.x), y = df_split1(r.y);
        reinterpret_cast<float4 *>(outv)[o + c * n] = make_float4(x.x, y.x, x.y, y.y);
      } else {
        out[o + c * n] = r;
      }
    }
  }
  if (MODE == 2 && part) {  // column sums over the CTA's sites (fixed order)
    double *red = reinterpret_cast<double *>(smem_raw);
#pragma unroll
    for (int off = IW; off < 32; off <<= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, off);
    __syncthreads();
    if (quad == 0) red[item] = nrm;
    __syncthreads();
    if (tid < n) {
      double sum = 0.0;
      for (int q = 0; q < nsites; ++q) sum += red[q * n + tid];
      part[(long)blockIdx.x * n + tid] = sum;
    }
  }
}

// out[p * n + c] = sum of the rows p, p + gridDim.x, ... of part (nblk x n), fixed order
__global__ void __launch_bounds__(256) k_fold_parts(const double *__restrict__ part, int nblk, int n,
                                                    double *__restrict__ out) {
  __shared__ double red[256];
  const int t = threadIdx.x, per = 256 / n, c = t % n, q0 = t / n;
  double s = 0.0;
  if (q0 < per)
    for (long r = (long)blockIdx.x + (long)q0 * gridDim.x; r < nblk; r += (long)per * gridDim.x) s += part[r * n + c];
  red[t] = s;
  __syncthreads();
  if (t < n) {
    double sum = 0.0;
    for (int q = 0; q < per; ++q) sum += red[q * n + t];
    out[(long)blockIdx.x * n + t] = sum;
  }
}

// Lanes per (site, right-hand side): four up to two warps per scheduler (four schedulers on
// each of 152 SMs), else one.  Sites per CTA: up to 128 threads, but at least a warp's
// worth while that gives the SMs more than two CTAs each, and at most 32 link records.
static int fx_split(const Geom &g, int n) { return g.Vh * n <= 2L * 4 * 152 * 32 ? 4 : 1; }
static int fx_tile(const Geom &g, int n, int split) {
  const int items = 128 / split;
  const int least = std::max(1, items / 4 / n);
  int tile = std::max(std::min(items / n, 32), least);
  while (tile > least && (g.Vh + tile - 1) / tile < 2 * 152) tile = std::max(least, tile / 2);
  return tile;
}

size_t hop_fx_conv_bytes(const Geom &g, int n) {
  return fx_split(g, n) == 4 ? 0 : (size_t)g.Vh * n * (3 * sizeof(int4) + sizeof(int));
}

long hop_fx_parts(const Geom &g, int n) {
  const int tile = fx_tile(g, n, fx_split(g, n));
  return (g.Vh + tile - 1) / tile;
}

// in64: the input in FP64; the four-lane kernel converts it itself, else it is
// converted into `in` first.  A lone FP64 hop (MODE 0) without a buffer for that takes the
// four-lane kernel on every lattice (24^4, n = 16: 913 us; with the conversion 393 us).
template <int MODE>
static rhmc_status_t launch_hop_fx(const Geom &g, int par, const FxLinks &L, const double2 *in64, FxField in,
                                   void *out, int *oex, const double2 *self, double a, int n, const double2 *B,
                                   float2 *outf, double *part, int cat, cudaStream_t s) {
  if (n < 1 || n > RHMC_MAX_NRHS || g.Vh * 3L * n > 0x7fffffffL) return RHMC_ERR_INVALID_ARG;
  const int split = MODE == 0 && !in.v ? 4 : fx_split(g, n), iw = 32 / split;
  if (in64 && split == 1) RHMC_TRY(fx_convert(g, in64, in, n, s));
  const int tile = fx_tile(g, n, split);
  const int threads = (tile * n + iw - 1) / iw * 32;
  const size_t smem = (size_t)tile * (73 * sizeof(int4) + 8 * sizeof(int));
  const unsigned grid = (unsigned)((g.Vh + tile - 1) / tile);
  prof_begin(cat, s);
  auto run = [&](auto kern) {
    kern<<<grid, threads, smem, s>>>(g, par, L.rec, L.exp, L.l64, in.v, in.e, in64, out, oex, self, a, n, tile, B, outf,
                                     part);
  };
  constexpr bool kFrom64 = MODE == 0 || MODE == 3 || MODE == 4;  // (these are always given in64, the others never)
  if (split == 4)
    run(k_hop_fx<MODE, 4, kFrom64>);
  else
    run(k_hop_fx<MODE, 1, false>);
  // algorithmic bytes: every link once, the inputs once, the outputs once
  const double fields = 2.0 + (MODE == 1 ? 1.0 : 0.0) + (MODE == 2 ? 2.0 + (outf ? 0.5 : 0.0) : 0.0);
  prof_end(s, (double)g.Vh * 16 * (72.0 + 3.0 * n * fields));
  RHMC_LAUNCH_CHECK();
  return RHMC_OK;
}

rhmc_status_t hop_fx(const Geom &g, int par, const FxLinks &L, const double2 *in, FxField conv, FxField out, int n,
                     int cat, cudaStream_t s) {
  return launch_hop_fx<4>(g, par, L, in, conv, out.v, out.e, nullptr, 0.0, n, nullptr, nullptr, nullptr, cat, s);
}

rhmc_status_t hop_fx_to64(const Geom &g, int par, const FxLinks &L, const double2 *in, FxField conv, double2 *out,
                          int n, cudaStream_t s) {
  return launch_hop_fx<0>(g, par, L, in, conv, out, nullptr, nullptr, 0.0, n, nullptr, nullptr, nullptr, PROF_HOP64, s);
}

rhmc_status_t hop_fx_self(const Geom &g, int par, const FxLinks &L, FxField in, double2 *out, const double2 *self,
                          double a, int n, cudaStream_t s) {
  return launch_hop_fx<1>(g, par, L, nullptr, in, out, nullptr, self, a, n, nullptr, nullptr, nullptr, PROF_HOP64, s);
}

rhmc_status_t hop_fx_to_df(const Geom &g, int par, const FxLinks &L, const double2 *in, FxField conv, float4 *out,
                           int n, cudaStream_t s) {
  return launch_hop_fx<3>(g, par, L, in, conv, out, nullptr, nullptr, 0.0, n, nullptr, nullptr, nullptr, PROF_HOP_DF,
                          s);
}

rhmc_status_t resid_fx(const Geom &g, const FxLinks &L, FxField tmp, const double2 *X, double a, const double2 *B,
                       double2 *R, float2 *Rf, int n, double *scratch, double *part, int nparts, cudaStream_t s) {
  RHMC_TRY(launch_hop_fx<2>(g, 0, L, nullptr, tmp, R, nullptr, X, a, n, B, Rf, part ? scratch : nullptr, PROF_HOP_DF, s));
  if (part) {
    k_fold_parts<<<nparts, 256, 0, s>>>(scratch, (int)hop_fx_parts(g, n), n, part);
    RHMC_LAUNCH_CHECK();
  }
  return RHMC_OK;
}

// FP64 -> double-float pairs of complex fields (the force kernel's operands).
__global__ void k_df_convert(const double2 *__restrict__ in64, float4 *__restrict__ outdf, long len) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= len) return;
  const double2 z = in64[i];
  const float2 a = df_split1(z.x), b = df_split1(z.y);
  outdf[i] = make_float4(a.x, b.x, a.y, b.y);
}

rhmc_status_t df_split(const double2 *in, float4 *out, long len, cudaStream_t s) {
  k_df_convert<<<(unsigned)((len + 255) / 256), 256, 0, s>>>(in, out, len);
  RHMC_LAUNCH_CHECK();
  return RHMC_OK;
}

template rhmc_status_t hop<float>(const Geom &, int, const float2 *, const float2 *, float2 *, const float2 *, double,
                                  int, int, long, cudaStream_t, const float2 *, int, const SolverState *);
template rhmc_status_t hop<double>(const Geom &, int, const double2 *, const double2 *, double2 *, const double2 *,
                                   double, int, int, long, cudaStream_t, const double2 *, int, const SolverState *);

// 12-real copies of the FP32 records; returns through *ok whether every record
// is f V with V in SU(3) to FP32 accuracy (then the hop may use the copies).
rhmc_status_t stage_links12(const Geom &g, int bc_t, float2 *const l32[2], float2 *l12[2], bool *ok,
                            cudaStream_t s) {
  unsigned *dmax = nullptr;
  RHMC_CUDA_TRY(cudaMallocAsync(&dmax, sizeof(unsigned), s));
  RHMC_CUDA_TRY(cudaMemsetAsync(dmax, 0, sizeof(unsigned), s));
  const long items = g.Vh * 8;
  for (int p = 0; p < 2; ++p) {
    k_links12<<<(unsigned)((items + 255) / 256), 256, 0, s>>>(g, p, bc_t, l32[p], l12[p], dmax);
    RHMC_LAUNCH_CHECK();
  }
  unsigned h = 0;
  RHMC_CUDA_TRY(cudaMemcpyAsync(&h, dmax, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  RHMC_CUDA_TRY(cudaStreamSynchronize(s));
  RHMC_CUDA_TRY(cudaFreeAsync(dmax, s));
  float dev = 0.f;
  std::memcpy(&dev, &h, sizeof(float));
  *ok = dev < 1e-5f;
  return RHMC_OK;
}

}  // namespace rhmc
