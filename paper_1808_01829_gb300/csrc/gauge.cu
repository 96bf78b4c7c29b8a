// The RHMC trajectory around the pseudofermion force (Sec. II set-up; Sec. IV
// run parameters: Wilson gauge action, two-level OMF2 integrator, heatbath and
// accept/reject with 1e-14 solves).  FP64 throughout: next to the force solves
// these kernels are a few percent of a trajectory.
//
// Conventions (the force's):
//   * U[site][mu][3][3], site = x + Lx (y + Ly (z + Lz t)), periodic links;
//   * S_g = beta sum_{x, mu<nu} (1 - Re tr Pi_{mu nu}(x) / 3),
//     Pi_{mu nu}(x) = U_mu(x) U_nu(x+mu) U_mu(x+nu)^dagger U_nu(x)^dagger;
//   * G = dS/dRe U + i dS/dIm U; the plaquettes through U_mu(x) add up to
//     Re tr(U_mu(x) V_mu(x)) with the staple sum
//     V_mu(x) = sum_{nu != mu} [U_nu(x+mu) U_mu(x+nu)^dagger U_nu(x)^dagger
//                              + U_nu(x+mu-nu)^dagger U_mu(x-nu)^dagger U_nu(x-nu)],
//     so G_g = -(beta / 3) V^dagger;
//   * P = sum_a p^a T^a (T^a = i lambda^a / 2), dU/dtau = P U,
//     K = -sum tr(P^2) = sum_a (p^a)^2 / 2, dP/dtau = TA(U G^dagger) / 2,
//     TA(M) = (M - M^dagger)/2 - tr(M - M^dagger)/6.
// One thread per link (or site, for the plaquettes); the reductions write one
// partial sum per CTA, added on the host in a fixed order.
#include <cmath>
#include <vector>

#include "common.cuh"
#include "fx.cuh"
#include "kernels.h"

namespace rhmc {

namespace {
constexpr int kTaylor = 16;  // degree of the exponential's Taylor polynomial (argument norm <= 1/2)

struct M3 {
  double2 e[9];
};

__device__ __forceinline__ M3 ld3(const double2 *p) {
  M3 m;
#pragma unroll
  for (int k = 0; k < 9; ++k) m.e[k] = p[k];
  return m;
}
__device__ __forceinline__ M3 zero3() {
  M3 m;
#pragma unroll
  for (int k = 0; k < 9; ++k) m.e[k] = make_double2(0.0, 0.0);
  return m;
}
// a b
__device__ __forceinline__ M3 mul(const M3 &a, const M3 &b) {
  M3 c;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double re = 0.0, im = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double2 x = a.e[i * 3 + k], y = b.e[k * 3 + j];
        re = fma(x.x, y.x, fma(-x.y, y.y, re));
        im = fma(x.x, y.y, fma(x.y, y.x, im));
      }
      c.e[i * 3 + j] = make_double2(re, im);
    }
  return c;
}
// a b^dagger
__device__ __forceinline__ M3 mul_nd(const M3 &a, const M3 &b) {
  M3 c;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double re = 0.0, im = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double2 x = a.e[i * 3 + k], y = b.e[j * 3 + k];  // x conj(y)
        re = fma(x.x, y.x, fma(x.y, y.y, re));
        im = fma(x.y, y.x, fma(-x.x, y.y, im));
      }
      c.e[i * 3 + j] = make_double2(re, im);
    }
  return c;
}
// a^dagger b
__device__ __forceinline__ M3 mul_dn(const M3 &a, const M3 &b) {
  M3 c;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      double re = 0.0, im = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double2 x = a.e[k * 3 + i], y = b.e[k * 3 + j];  // conj(x) y
        re = fma(x.x, y.x, fma(x.y, y.y, re));
        im = fma(x.x, y.y, fma(-x.y, y.x, im));
      }
      c.e[i * 3 + j] = make_double2(re, im);
    }
  return c;
}
__device__ __forceinline__ void addto(M3 &a, const M3 &b) {
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    a.e[k].x += b.e[k].x;
    a.e[k].y += b.e[k].y;
  }
}
// p += c TA(m)
__device__ __forceinline__ void add_ta(double2 *p, const M3 &m, double c) {
  const double t = (m.e[0].y + m.e[4].y + m.e[8].y) / 3.0;  // Im tr(M) / 3: (M - M^dagger)/2 has an imaginary diagonal
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const double2 a = m.e[i * 3 + j], b = m.e[j * 3 + i];
      double2 f = make_double2(0.5 * (a.x - b.x), 0.5 * (a.y + b.y));
      if (i == j) f.y -= t;
      double2 q = p[i * 3 + j];
      q.x = fma(c, f.x, q.x);
      q.y = fma(c, f.y, q.y);
      p[i * 3 + j] = q;
    }
}

__device__ __forceinline__ void lex_coords(const Geom &g, long lex, int x[4]) {
  long r = lex;
  x[0] = (int)(r % g.L[0]);
  r /= g.L[0];
  x[1] = (int)(r % g.L[1]);
  r /= g.L[1];
  x[2] = (int)(r % g.L[2]);
  x[3] = (int)(r / g.L[2]);
}
// x + d mu (periodic), d = +1 / -1, as coordinates
__device__ __forceinline__ void step(const Geom &g, const int x[4], int mu, int d, int y[4]) {
#pragma unroll
  for (int nu = 0; nu < 4; ++nu) {
    int v = x[nu];
    if (nu == mu) {
      v += d;
      if (v < 0) v += g.L[nu];
      if (v >= g.L[nu]) v -= g.L[nu];
    }
    y[nu] = v;
  }
}
__device__ __forceinline__ M3 link(const double2 *U, const Geom &g, const int x[4], int mu) {
  return ld3(U + (lex_of(g, x) * 4 + mu) * 9);
}

// sum of the partial sums of a CTA (blockDim.x == 256) into partial[blockIdx.x]
__device__ __forceinline__ void cta_sum(double v, double *partial) {
  __shared__ double red[256];
  red[threadIdx.x] = v;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = red[0];
}
}  // namespace

// partial[b] = sum over the CTA's sites and planes mu < nu of (1 - Re tr Pi / 3).
// Re tr(A B^dagger) = sum_ij Re(A_ij conj(B_ij)) with A = U_mu(x) U_nu(x+mu),
// B = U_nu(x) U_mu(x+nu).
__global__ void __launch_bounds__(256) k_plaquette(Geom g, const double2 *__restrict__ U, double *__restrict__ partial) {
  double acc = 0.0;
  for (long site = (long)blockIdx.x * blockDim.x + threadIdx.x; site < g.V; site += (long)gridDim.x * blockDim.x) {
    int x[4];
    lex_coords(g, site, x);
    for (int mu = 0; mu < 3; ++mu) {
      int xm[4];
      step(g, x, mu, 1, xm);
      const M3 Um = ld3(U + (site * 4 + mu) * 9);
      for (int nu = mu + 1; nu < 4; ++nu) {
        int xn[4];
        step(g, x, nu, 1, xn);
        const M3 A = mul(Um, link(U, g, xm, nu));
        const M3 B = mul(ld3(U + (site * 4 + nu) * 9), link(U, g, xn, mu));
        double rt = 0.0;
#pragma unroll
        for (int k = 0; k < 9; ++k) rt = fma(A.e[k].x, B.e[k].x, fma(A.e[k].y, B.e[k].y, rt));
        acc += 1.0 - rt / 3.0;
      }
    }
  }
  cta_sum(acc, partial);
}

// partial[b] = -sum over the CTA's links of Re tr(P P)
__global__ void __launch_bounds__(256) k_kinetic(const double2 *__restrict__ P, long nlinks, double *__restrict__ partial) {
  double acc = 0.0;
  for (long l = (long)blockIdx.x * blockDim.x + threadIdx.x; l < nlinks; l += (long)gridDim.x * blockDim.x) {
    const M3 p = ld3(P + l * 9);
    double rt = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const double2 a = p.e[i * 3 + j], b = p.e[j * 3 + i];
        rt = fma(a.x, b.x, fma(-a.y, b.y, rt));
      }
    acc -= rt;
  }
  cta_sum(acc, partial);
}

// P = sum_a p^a T^a, T^a = i lambda^a / 2 in the standard Gell-Mann basis
__global__ void __launch_bounds__(256) k_momenta(const double *__restrict__ p, double2 *__restrict__ P, long nlinks) {
  const long l = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= nlinks) return;
  double a[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) a[k] = 0.5 * p[l * 8 + k];
  const double r3 = 0.57735026918962576451;  // 1 / sqrt(3)
  double2 *o = P + l * 9;
  o[0] = make_double2(0.0, a[2] + r3 * a[7]);
  o[4] = make_double2(0.0, -a[2] + r3 * a[7]);
  o[8] = make_double2(0.0, -2.0 * r3 * a[7]);
  o[1] = make_double2(a[1], a[0]);   // i (lambda1 p1 + lambda2 p2) / 2, entry (0, 1)
  o[3] = make_double2(-a[1], a[0]);  // entry (1, 0)
  o[2] = make_double2(a[4], a[3]);
  o[6] = make_double2(-a[4], a[3]);
  o[5] = make_double2(a[6], a[5]);
  o[7] = make_double2(-a[6], a[5]);
}

// P_mu(x) += coef TA(U_mu(x) V_mu(x)); the kick P += eps TA(U G_g^dagger)/2 with
// G_g = -(beta/3) V^dagger has coef = -eps beta / 6.  FP64 form, one link e.
__device__ __noinline__ void kick_fp64(const Geom &g, const double2 *U, double2 *P, double coef, long e) {
  const long site = e >> 2;
  const int mu = (int)(e & 3);
  int x[4], xp[4];
  lex_coords(g, site, x);
  step(g, x, mu, 1, xp);
  M3 V = zero3();
  for (int nu = 0; nu < 4; ++nu) {
    if (nu == mu) continue;
    int xn[4], xd[4], xpd[4];
    step(g, x, nu, 1, xn);   // x + nu
    step(g, x, nu, -1, xd);  // x - nu
    step(g, xd, mu, 1, xpd); // x + mu - nu
    // U_nu(x+mu) U_mu(x+nu)^dagger U_nu(x)^dagger
    addto(V, mul_nd(mul_nd(link(U, g, xp, nu), link(U, g, xn, mu)), ld3(U + (site * 4 + nu) * 9)));
    // (U_mu(x-nu) U_nu(x+mu-nu))^dagger U_nu(x-nu)
    addto(V, mul_dn(mul(link(U, g, xd, mu), link(U, g, xpd, nu)), link(U, g, xd, nu)));
  }
  add_ta(P + e * 9, mul(ld3(U + e * 9), V), coef);
}

// The same for one link by all 32 lanes of a warp: lane 9 s + 3 i + j forms entry (i, j) of the two
// staples of the s-th direction and of U V, the factors' rows by shuffles.  About 3 us, where a
// lane on its own takes 45.
__device__ __noinline__ void kick_fp64_warp(const Geom &g, const double2 *U, double2 *P, double coef, long site,
                                            int mu) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31, s = lane / 9, e = lane - 9 * s, i = e / 3, j = e - 3 * i;
  const int nu = s == 3 ? (mu ? 0 : 1) : s < mu ? s : s + 1;  // (lanes 27 to 31 only take part in the shuffles)
  int x[4], xp[4], xn[4], xd[4], xpd[4];
  lex_coords(g, site, x);
  step(g, x, mu, 1, xp);
  step(g, x, nu, 1, xn);
  step(g, x, nu, -1, xd);
  step(g, xd, mu, 1, xpd);
  const double2 *un = U + (site * 4 + nu) * 9, *up = U + (lex_of(g, xp) * 4 + nu) * 9,
                *mn = U + (lex_of(g, xn) * 4 + mu) * 9, *md = U + (lex_of(g, xd) * 4 + mu) * 9,
                *pd = U + (lex_of(g, xpd) * 4 + nu) * 9, *nd = U + (lex_of(g, xd) * 4 + nu) * 9;
  auto from = [&](double2 z, int src) {
    return make_double2(__shfl_sync(kAll, z.x, src & 31), __shfl_sync(kAll, z.y, src & 31));
  };
  auto conj = [](double2 z) { return make_double2(z.x, -z.y); };
  double2 a = make_double2(0.0, 0.0), b = a, f = a, h = a;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    cmac<double>(a, up[i * 3 + k], conj(mn[j * 3 + k]));  // U_nu(x+mu) U_mu(x+nu)^dagger
    cmac<double>(b, md[i * 3 + k], pd[k * 3 + j]);        // U_mu(x-nu) U_nu(x+mu-nu)
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    cmac<double>(f, from(a, 9 * s + 3 * i + k), conj(un[j * 3 + k]));
    cmac<double>(h, conj(from(b, 9 * s + 3 * k + i)), nd[k * 3 + j]);
  }
  const double2 v = make_double2(f.x + h.x, f.y + h.y);
  const double2 v0 = from(v, e), v1 = from(v, 9 + e), v2 = from(v, 18 + e);
  const double2 V = make_double2(v0.x + v1.x + v2.x, v0.y + v1.y + v2.y);
  double2 w = make_double2(0.0, 0.0);
#pragma unroll
  for (int k = 0; k < 3; ++k) cmac<double>(w, U[(site * 4 + mu) * 9 + i * 3 + k], from(V, 3 * k + j));
  const double2 t = from(w, 3 * j + i);
  const double tr = (from(w, 0).y + from(w, 4).y + from(w, 8).y) / 3.0;
  if (lane < 9) {
    double2 *p = P + (site * 4 + mu) * 9 + e;
    const double2 z = *p;
    *p = make_double2(fma(coef, 0.5 * (w.x - t.x), z.x),
                      fma(coef, 0.5 * (w.y + t.y) - (i == j ? tr : 0.0), z.y));
  }
}

__global__ void __launch_bounds__(128) k_gauge_momentum(Geom g, const double2 *__restrict__ U, double2 *__restrict__ P,
                                                        double coef) {
  const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < 4 * g.V) kick_fp64(g, U, P, coef, e);
}

// ------------------------------------------------------------ the kick on the integer units
namespace {
// |r| <= most
__device__ __forceinline__ bool within(long long r, long long most) {
  return (unsigned long long)(r + most) <= 2ull * most;
}
// Largest entry of a link and of a product (one, to rounding) and largest staple sum (eight): sums
// of the two high words of a complex stay within 2^29 + 2^14, 2^30 + 2^15 and 2^31 - 2 (a value
// rounds up to the next high word within 2^26 of it), and sums of three products below 2^62.
constexpr long long kMostLink = (1ll << 55) + (1ll << 40), kMostProduct = (1ll << 56) + (1ll << 41),
                    kMostStaples = (1ll << 57) - (1ll << 26) - 1;
}  // namespace

// The 13 products of 3 x 3 matrices of a link's kick (1404 FP64 FMAs, 64 clocks each for a
// warp) as exact integer sums (fx.cuh): 243 multiply-adds of four clocks per product.  The
// entries of SU(3) links, their products and the sum of six staples have known sizes, so
// links are held in units of 2^-55, products of two in 2^-56, staples in 2^-57 and their sum in
// 2^-54 (two words, hi 2^27 + lo), and a product needs no shift: 2^-54 of it is
// h1 h2 + (h1 l2 + l1 h2) 2^-27 + l1 l2 2^-54, the last term dropped.
// Links whose largest entry is not in [1/4, 1] (to rounding), products above that and staple
// sums of 8 or more (never for SU(3)) send the link's kick to the FP64 form.
// So does a kick whose FP64 form would be more accurate than these units: its rounding is
// relative to the sizes of the products that form an entry, sum_k |U_ik| |V_kj|, which is small
// next to one for links near the unit matrix (weak fields) or near a block form.
// The links are converted once, to v[(mu * 9 + entry) * V + site], so that the warps of the
// kick, 32 consecutive sites of one direction each, read whole lines; ok[mu * V + site] says
// whether the link fits (kFits) and whether it is near a real diagonal matrix (kWeak).
constexpr int kFits = 1, kWeak = 2;
__global__ void __launch_bounds__(128) k_links_to_fx(const double2 *__restrict__ U, int4 *__restrict__ v,
                                                     int *__restrict__ ok, long V) {
  const int mu = threadIdx.x >> 5;
  const long site = (long)blockIdx.x * 32 + (threadIdx.x & 31);
  if (site >= V) return;
  const M3 u = ld3(U + (site * 4 + mu) * 9);
  int ef = 0, small = 0;  // largest exponent field, and that of all but the real diagonal
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    const int re = fx::expo(u.e[c].x), im = fx::expo(u.e[c].y);
    ef = max(ef, max(re, im));
    small = max(small, max(c % 4 ? re : 0, im));
  }
  bool fits = ef >= 1021 && ef <= 1023;
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    const long long qr = fits ? fx::fixed55(u.e[c].x) : 0, qi = fits ? fx::fixed55(u.e[c].y) : 0;
    fits = fits && within(qr, kMostLink) && within(qi, kMostLink);
    const int2 re = fx::words(qr), im = fx::words(qi);
    v[(mu * 9 + c) * V + site] = make_int4(re.x, re.y, im.x, im.y);
  }
  ok[mu * V + site] = (fits ? kFits : 0) | (small < 1023 - 6 ? kWeak : 0);
}

namespace {
// three sums r_j = sum_k a_k b[k][j] in a_k's and b's units multiplied by 2^54, rounded (re, im)
__device__ __forceinline__ void row_times(const int4 *a, const int4 *b, long long *r) {
  constexpr long long half = 1ll << (fx::kLow - 1);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    long long pA = 0, pB = half, mA = 0, mB = 0, iA = 0, iB = 2 * half;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int4 x = a[k], y = b[k * 3 + j];
      fx::mac2(pA, pB, x.x, x.y, y.x, y.y);
      fx::mac2(mA, mB, x.z, x.w, y.z, y.w);
      fx::mac2(iA, iB, x.x + x.z, x.y + x.w, y.x + y.z, y.y + y.w);
    }
    r[2 * j] = fx::join(pA - mA, pB - mB);
    r[2 * j + 1] = fx::join(iA - pA - mA, iB - pB - mB);
  }
}
// Sizes (in units of 2^-20) below which the FP64 form is the more accurate one; see k_gauge_momentum_fx
constexpr int kOffSize = (int)(0.8 * (1 << 20)), kDiagSize = (int)(0.4 * (1 << 20));
// Links of a warp that need the FP64 form: up to this many one by one with all lanes
constexpr int kFew = 12;
__device__ __forceinline__ int4 conj_if(int4 z, int m) {  // m = -1: the conjugate, 0: z
  return make_int4(z.x, z.y, (z.z ^ m) - m, (z.w ^ m) - m);
}
// p += coef TA(w) for w in units of 2^-55
__device__ __forceinline__ void add_ta_fx(double2 *p, const long long *w, double coef) {
  // TA(w) = (w - w^dagger)/2 - tr(w - w^dagger)/6; its upper triangle, twice as large
  const long long tr = (w[1] + w[9] + w[17]) / 3;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const double d = fx::value(w[2 * (i * 4) + 1] - tr, -54);
    double2 z = p[i * 4];
    z.y = fma(0.5 * coef, d, z.y);
    p[i * 4] = z;
#pragma unroll
    for (int j = i + 1; j < 3; ++j) {
      const int a = 2 * (i * 3 + j), c = 2 * (j * 3 + i);
      const double re = fx::value(w[a] - w[c], -55), im = fx::value(w[a + 1] + w[c + 1], -55);
      double2 z1 = p[i * 3 + j], z2 = p[j * 3 + i];
      z1.x = fma(0.5 * coef, re, z1.x);
      z1.y = fma(0.5 * coef, im, z1.y);
      z2.x = fma(-0.5 * coef, re, z2.x);
      z2.y = fma(0.5 * coef, im, z2.y);
      p[i * 3 + j] = z1;
      p[j * 3 + i] = z2;
    }
  }
}
}  // namespace

// The kick of k_gauge_momentum with integer products.  A staple is op(X) Y^dagger op'(Z)
// (forward: X, Z^dagger; backward: X^dagger, Z), formed row by row; the six are added as
// integers and only the traceless anti-Hermitian part of U V is converted to FP64.
// The loops over staples and rows are not unrolled, and the sum lives in shared memory:
// unrolled, the warps waited for instructions.  Bound by the integer multiplier, 13 x 243
// multiply-adds of four clocks per link (175 us at 16^3 x 32), and by the adds and shifts around
// them at two warps per scheduler.  Measured at 16^3 x 32, with the conversion: 568 us, 1795 us in
// FP64.  Error of the force (largest entry, relative to the largest of the lattice): links
// exp(i eps H) with eps = 0.5 8.1e-17, FP64 form 2.3e-16.
// The error in these units is the same for every link, that of the FP64 form is relative to
// S_ij = sum_k |U_ik| |V_kj| + |U_jk| |V_ki| off the diagonal and to the largest of
// sum_k |Re U_ik| |Im V_ki| + |Im U_ik| |Re V_ki| on it.  They meet where these are 0.8 and 0.4
// (both forms up to 1.6e-16 S and 4.4e-16 S); a link below either takes the FP64 form, a few
// of a warp with all its lanes, many each with its own.  At eps = 0.5 no link does, at 0.3
// one in 2000 (573 us; 660 us with a lane each), at 0.2 646 us (1220), 1.46 ms at 0.1, at most 1.78 ms.
__global__ void __launch_bounds__(128, 2) k_gauge_momentum_fx(Geom g, const int4 *__restrict__ v,
                                                              const int *__restrict__ ok,
                                                              const double2 *__restrict__ U, double2 *__restrict__ P,
                                                              double coef) {
  __shared__ long long sV[18][128];  // the staple sum V of this thread
  const int mu = threadIdx.x >> 5, tid = threadIdx.x;
  const int nsite = (int)g.V, site = blockIdx.x * 32 + (threadIdx.x & 31);
  if (site >= nsite) return;
#pragma unroll
  for (int c = 0; c < 18; ++c) sV[c][tid] = 0;
  int x[4], xp[4];
  {
    int r = site;
    x[0] = r % g.L[0];
    r /= g.L[0];
    x[1] = r % g.L[1];
    r /= g.L[1];
    x[2] = r % g.L[2];
    x[3] = r / g.L[2];
  }
  step(g, x, mu, 1, xp);
  const int sp = (int)lex_of(g, xp);
  const bool whole = blockIdx.x * 32 + 32 <= nsite;  // every lane of the CTA has a site
  const int flags = ok[mu * nsite + site];
  bool fits = flags & kFits;
#pragma unroll 1
  for (int q = 0; q < 6; ++q) {
    const int nu = (q >> 1) < mu ? (q >> 1) : (q >> 1) + 1;
    const bool fwd = (q & 1) == 0;
    int xn[4], xq[4];
    step(g, x, nu, fwd ? 1 : -1, xn);
    step(g, xn, mu, 1, xq);
    const int sn = (int)lex_of(g, xn);
    const int sx = fwd ? sp : (int)lex_of(g, xq), sz = fwd ? site : sn;
    const int near = flags & ok[nu * nsite + sx] & ok[mu * nsite + sn] & ok[nu * nsite + sz];
    fits = fits && (near & kFits);
    // a warp with many such plaquettes: the FP64 form will be needed at the end, so at once
    if (q == 0 && (whole ? __popc(__ballot_sync(0xffffffffu, near & kWeak)) > kFew : near & kWeak)) {
      kick_fp64(g, U, P, coef, (long)site * 4 + mu);
      return;
    }
    const int4 *px = v + (long)nu * 9 * nsite + sx, *py = v + (long)mu * 9 * nsite + sn,
               *pz = v + (long)nu * 9 * nsite + sz;
    const int cz = fwd ? -1 : 0;
    const int rs = fwd ? 3 : 1, cs = fwd ? 1 : 3;  // strides of op(X)'s rows and columns
    int4 y[9], z[9];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        y[k * 3 + j] = conj_if(__ldg(py + (j * 3 + k) * nsite), -1);
        z[k * 3 + j] = conj_if(__ldg(pz + (j * rs + k * cs) * nsite), cz);
      }
#pragma unroll 1
    for (int i = 0; i < 3; ++i) {
      int4 a[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) a[k] = conj_if(__ldg(px + (i * rs + k * cs) * nsite), ~cz);
      long long r[6];
      row_times(a, y, r);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        fits = fits && within(r[2 * k], kMostProduct) && within(r[2 * k + 1], kMostProduct);
        const int2 re = fx::words(r[2 * k]), im = fx::words(r[2 * k + 1]);
        a[k] = make_int4(re.x, re.y, im.x, im.y);
      }
      row_times(a, z, r);
#pragma unroll
      for (int c = 0; c < 6; ++c) sV[i * 6 + c][tid] += r[c];
    }
  }
  int4 b[9];
  int vr[9], vi[9];  // sizes of the parts of V in units of 2^-10
#pragma unroll
  for (int c = 0; c < 9; ++c) {
    const long long re = (sV[2 * c][tid] + 4) >> 3, im = (sV[2 * c + 1][tid] + 4) >> 3;
    fits = fits && within(re, kMostStaples) && within(im, kMostStaples);
    const int2 wr = fx::words(re), wi = fx::words(im);
    b[c] = make_int4(wr.x, wr.y, wi.x, wi.y);
    vr[c] = abs(wr.x) >> 17;
    vi[c] = abs(wi.x) >> 17;
  }
  long long w[18];
  int od[3] = {0, 0, 0}, di = 0;  // sum_k |U_ik| |V_kj| + |U_jk| |V_ki|, and that of the diagonal's imaginary part
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    int4 a[3];
    int d = 0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      a[c] = __ldg(v + (long)(mu * 9 + i * 3 + c) * nsite + site);
      const int ur = abs(a[c].x) >> 18, ui = abs(a[c].z) >> 18;  // (units of 2^-10)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        if (j != i) od[i + j - 1] += (ur + ui) * (vr[c * 3 + j] + vi[c * 3 + j]);
      d += ur * vi[c * 3 + i] + ui * vr[c * 3 + i];
    }
    di = max(di, d);
    row_times(a, b, w + 6 * i);
  }
  const bool fp64 = !fits || min(od[0], min(od[1], od[2])) < kOffSize || di < kDiagSize;
  if (!fp64) add_ta_fx(P + ((long)site * 4 + mu) * 9, w, coef);
  unsigned left = whole ? __ballot_sync(0xffffffffu, fp64) : 0u;
  if (!whole || __popc(left) > kFew) {
    if (fp64) kick_fp64(g, U, P, coef, (long)site * 4 + mu);
  } else {
    for (; left; left &= left - 1) kick_fp64_warp(g, U, P, coef, (long)blockIdx.x * 32 + __ffs(left) - 1, mu);
  }
}

// P += coef TA(U G^dagger)
__global__ void __launch_bounds__(128) k_momentum_update(const double2 *__restrict__ U, const double2 *__restrict__ G,
                                                         double2 *__restrict__ P, long nlinks, double coef) {
  const long l = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= nlinks) return;
  add_ta(P + l * 9, mul_nd(ld3(U + l * 9), ld3(G + l * 9)), coef);
}

// U <- exp(Y) U, Y = eps P.  exp(Y) for |Y|_F <= 1/2 by its Taylor polynomial; larger
// arguments are scaled by 2^-k first and the result squared k times.  With the
// Cayley-Hamilton identity P^3 = t P^2 - s P + d (t = tr P, s = (t^2 - tr P^2) / 2, d = det P)
// the polynomial is f_0 + f_1 Y + f_2 Y^2, and its Horner steps act on three complex numbers:
//   (f_0, f_1, f_2) <- (1 + d f_2 / k, (f_0 - s f_2) / k, (f_1 + t f_2) / k)
// (t, s, d scaled by eps, eps^2, eps^3): 18 FP64 operations instead of the 126 of a matrix
// product, for any P.  exp(Y) - 1 = D is carried instead of exp(Y), so that U + D U rounds at
// the size of D.  The degree is the smallest whose remainder |Y|^(m+1) / (m+1)! e^|Y| is below
// 4e-20, the bound of degree 16 at |Y| = 1/2.  Bound by the FP64 pipe, about 500 operations per
// link.  Measured at 16^3 x 32: 508 us, 1922 us with matrix products at degree 16; against a
// 113-bit sum the error of U is 4e-17 at eps = 0.05 (7.7e-17 with matrix products).
__constant__ double kRecip[kTaylor + 1] = {0.0,      1.0,      1.0 / 2,  1.0 / 3,  1.0 / 4,  1.0 / 5,
                                           1.0 / 6,  1.0 / 7,  1.0 / 8,  1.0 / 9,  1.0 / 10, 1.0 / 11,
                                           1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15, 1.0 / 16};
__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 zscale(double2 a, double r) { return make_double2(a.x * r, a.y * r); }
__global__ void __launch_bounds__(128) k_link_update(double2 *__restrict__ U, const double2 *__restrict__ P, long nlinks,
                                                     double eps) {
  const long l = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= nlinks) return;
  M3 p = ld3(P + l * 9);
  auto norm2 = [&]() {
    double n = 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k) n = fma(p.e[k].x, p.e[k].x, fma(p.e[k].y, p.e[k].y, n));
    return n;
  };
  double n2 = norm2();
  int sq = 0;
  double sc = eps;
  if (n2 > 1e-100 && n2 < 1e100) {
    n2 *= eps * eps;
  } else {  // det P could leave the range of FP64 where Y = eps P does not
#pragma unroll
    for (int k = 0; k < 9; ++k) p.e[k] = zscale(p.e[k], eps);
    sc = 1.0;
    n2 = norm2();
  }
  while (n2 > 0.25 && sq < 64) {  // bounded: a non-finite norm stops at 64
    n2 *= 0.25;
    sc *= 0.5;
    ++sq;
  }
  int deg = 0;
  {
    // from an upper bound of |Y| (NaN takes the full degree)
    const float ny = sqrtf((float)n2) * 1.0001f;
    float r = ny * __expf(ny) * 1.01f;  // remainder of degree 0
    while (deg < kTaylor && !(r < 4e-20f)) {
      ++deg;
      r *= ny / (float)(deg + 1);
    }
    deg = max(2, deg);
  }
  const M3 p2 = mul(p, p);
  const double sc2 = sc * sc;
  double2 tr = make_double2(p.e[0].x + p.e[4].x + p.e[8].x, p.e[0].y + p.e[4].y + p.e[8].y);
  const double2 q2 = make_double2(p2.e[0].x + p2.e[4].x + p2.e[8].x, p2.e[0].y + p2.e[4].y + p2.e[8].y);
  const double2 t2 = zmul(tr, tr);
  const double2 s = make_double2(0.5 * sc2 * (t2.x - q2.x), 0.5 * sc2 * (t2.y - q2.y));
  // det P along the first row
  auto minor = [&](int a, int b, int c, int d) {
    const double2 u = zmul(p.e[a], p.e[d]), w = zmul(p.e[b], p.e[c]);
    return make_double2(u.x - w.x, u.y - w.y);
  };
  const double2 m0 = zmul(p.e[0], minor(4, 5, 7, 8)), m1 = zmul(p.e[1], minor(3, 5, 6, 8)),
                m2 = zmul(p.e[2], minor(3, 4, 6, 7));
  const double2 d = zscale(make_double2(m0.x - m1.x + m2.x, m0.y - m1.y + m2.y), sc * sc2);
  tr = zscale(tr, sc);
  double2 f0 = make_double2(0.0, 0.0), f1 = f0, f2 = f0;  // f0: less one
  for (int k = deg; k >= 1; --k) {
    const double r = kRecip[k];
    const double2 g2 = zscale(f2, r);
    const double2 h0 = zmul(d, g2), h1 = zmul(s, g2), h2 = zmul(tr, g2);
    f2 = make_double2(fma(f1.x, r, h2.x), fma(f1.y, r, h2.y));
    f1 = make_double2(fma(f0.x, r, r - h1.x), fma(f0.y, r, -h1.y));
    f0 = h0;
  }
  f1 = zscale(f1, sc);
  f2 = zscale(f2, sc2);
  M3 D;
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    double2 a = q % 4 == 0 ? f0 : make_double2(0.0, 0.0);
    cmac<double>(a, f2, p2.e[q]);
    cmac<double>(a, f1, p.e[q]);
    D.e[q] = a;
  }
  if (sq) {  // |Y| > 1/2: 1 + D itself, squared (an exponential of small entries keeps their relative accuracy)
    D.e[0].x += 1.0;
    D.e[4].x += 1.0;
    D.e[8].x += 1.0;
    for (int i = 0; i < sq; ++i) D = mul(D, D);
  }
  const M3 u = ld3(U + l * 9);
  const M3 w = mul(D, u);
#pragma unroll
  for (int k = 0; k < 9; ++k)
    U[l * 9 + k] = sq ? w.e[k] : make_double2(u.e[k].x + w.e[k].x, u.e[k].y + w.e[k].y);
}

// ------------------------------------------------------------ launch wrappers
namespace {
constexpr size_t kLinkBytes = 9 * sizeof(double2);

rhmc_status_t reduce_parts(double *parts, int nparts, cudaStream_t s, double *out) {
  std::vector<double> h(nparts);
  RHMC_CUDA_TRY(cudaMemcpyAsync(h.data(), parts, sizeof(double) * nparts, cudaMemcpyDeviceToHost, s));
  RHMC_CUDA_TRY(cudaStreamSynchronize(s));
  double sum = 0.0;
  for (int q = 0; q < nparts; ++q) sum += h[q];
  *out = sum;
  return RHMC_OK;
}

struct Lat {
  int device = 0;
  Geom g{};
};
rhmc_status_t lattice(rhmc_ctx_t *c, Lat *l) { return ctx_lattice(c, &l->device, &l->g); }
}  // namespace

rhmc_status_t gauge_action(rhmc_ctx_t *c, const Geom &g, const double2 *U, double beta, double *S, cudaStream_t s) {
  double *parts;
  int nparts;
  RHMC_TRY(ctx_partials(c, &parts, &nparts));
  prof_begin(PROF_OTHER, s);
  k_plaquette<<<nparts, 256, 0, s>>>(g, U, parts);
  prof_end(s, (double)g.V * 4 * kLinkBytes);
  RHMC_LAUNCH_CHECK();
  double sum = 0.0;
  RHMC_TRY(reduce_parts(parts, nparts, s, &sum));
  *S = beta * sum;
  return RHMC_OK;
}

rhmc_status_t kinetic_energy(rhmc_ctx_t *c, const Geom &g, const double2 *P, double *K, cudaStream_t s) {
  double *parts;
  int nparts;
  RHMC_TRY(ctx_partials(c, &parts, &nparts));
  prof_begin(PROF_OTHER, s);
  k_kinetic<<<nparts, 256, 0, s>>>(P, g.V * 4, parts);
  prof_end(s, (double)g.V * 4 * kLinkBytes);
  RHMC_LAUNCH_CHECK();
  return reduce_parts(parts, nparts, s, K);
}

rhmc_status_t momenta_from_normals(const Geom &g, const double *p, double2 *P, cudaStream_t s) {
  const long nl = g.V * 4;
  prof_begin(PROF_OTHER, s);
  k_momenta<<<(unsigned)((nl + 255) / 256), 256, 0, s>>>(p, P, nl);
  prof_end(s, (double)nl * (8 * sizeof(double) + kLinkBytes));
  RHMC_LAUNCH_CHECK();
  return RHMC_OK;
}

rhmc_status_t gauge_momentum(rhmc_ctx_t *c, const Geom &g, const double2 *U, double2 *P, double beta, double eps, cudaStream_t s) {
  const long nl = g.V * 4;
  const unsigned grid = (unsigned)((g.V + 31) / 32);  // 128 threads: four directions of 32 sites
  // The integer form needs the links in integer form, in a buffer of the context.  A stream
  // that is being captured, and one for which there is no memory, takes the FP64 kernel.
  int4 *v = ctx_links_fx_begin(c, s);
  int *ex = v ? (int *)(v + 36 * g.V) : nullptr;
  if (v) {
    prof_begin(PROF_OTHER, s);
    k_links_to_fx<<<grid, 128, 0, s>>>(U, v, ex, g.V);
    prof_end(s, (double)nl * 2 * kLinkBytes);
    RHMC_LAUNCH_CHECK();
  }
  prof_begin(PROF_OTHER, s);
  if (v)
    k_gauge_momentum_fx<<<grid, 128, 0, s>>>(g, v, ex, U, P, -eps * beta / 6.0);
  else
    k_gauge_momentum<<<(unsigned)((nl + 127) / 128), 128, 0, s>>>(g, U, P, -eps * beta / 6.0);
  prof_end(s, (double)nl * 3 * kLinkBytes);
  RHMC_LAUNCH_CHECK();
  return v ? ctx_links_fx_end(c, s) : RHMC_OK;
}

rhmc_status_t momentum_update(const Geom &g, const double2 *U, const double2 *G, double2 *P, double eps,
                              cudaStream_t s) {
  const long nl = g.V * 4;
  prof_begin(PROF_OTHER, s);
  k_momentum_update<<<(unsigned)((nl + 127) / 128), 128, 0, s>>>(U, G, P, nl, 0.5 * eps);
  prof_end(s, (double)nl * 4 * kLinkBytes);
  RHMC_LAUNCH_CHECK();
  return RHMC_OK;
}

rhmc_status_t link_update(const Geom &g, double2 *U, const double2 *P, double eps, cudaStream_t s) {
  const long nl = g.V * 4;
  prof_begin(PROF_OTHER, s);
  k_link_update<<<(unsigned)((nl + 127) / 128), 128, 0, s>>>(U, P, nl, eps);
  prof_end(s, (double)nl * 3 * kLinkBytes);
  RHMC_LAUNCH_CHECK();
  return RHMC_OK;
}

// ------------------------------------------------------------ integrator
namespace {
struct Md {
  rhmc_ctx_t *c;
  Geom g;
  double2 *U, *P, *G;
  const void *Phi;
  int n_pf;
  const rhmc_rational_t *md;
  const rhmc_md_params_t *p;
  rhmc_md_info_t *info;
  cudaStream_t s;

  rhmc_status_t fermion_kick(double eps) {
    if (!Phi || n_pf == 0 || eps == 0.0) return RHMC_OK;
    RHMC_TRY(rhmc_set_gauge(c, U, s));
    rhmc_info_t fi{};
    const rhmc_status_t st = rhmc_force(c, Phi, n_pf, md->alpha0, md->alpha, md->beta, md->n_shifts, p->tol_md,
                                        p->max_iter, p->precision_md, nullptr, G, nullptr, nullptr, &fi, s);
    info->force_evals += 1;
    info->solver_iters += fi.iters + fi.refine_iters;
    info->dirac_calls += fi.dirac_calls;
    if (fi.true_rel_resid_max > info->max_rel_resid) info->max_rel_resid = fi.true_rel_resid_max;
    if (st != RHMC_OK) return st;
    return momentum_update(g, U, G, P, eps, s);
  }
  rhmc_status_t gauge_kick(double eps) {
    info->gauge_force_evals += 1;
    return gauge_momentum(c, g, U, P, p->beta, eps, s);
  }
  // D(h): n_gauge OMF2 steps of the gauge force, the kicks at the same links merged
  rhmc_status_t drift(double h) {
    const double e = h / p->n_gauge, lam = p->lambda;
    RHMC_TRY(gauge_kick(lam * e));
    for (int i = 0; i < p->n_gauge; ++i) {
      RHMC_TRY(link_update(g, U, P, 0.5 * e, s));
      RHMC_TRY(gauge_kick((1.0 - 2.0 * lam) * e));
      RHMC_TRY(link_update(g, U, P, 0.5 * e, s));
      RHMC_TRY(gauge_kick(i + 1 < p->n_gauge ? 2.0 * lam * e : lam * e));
    }
    return RHMC_OK;
  }
  rhmc_status_t run() {
    const double e = p->tau / p->n_steps, lam = p->lambda;
    RHMC_TRY(fermion_kick(lam * e));
    for (int k = 0; k < p->n_steps; ++k) {
      RHMC_TRY(drift(0.5 * e));
      RHMC_TRY(fermion_kick((1.0 - 2.0 * lam) * e));
      RHMC_TRY(drift(0.5 * e));
      RHMC_TRY(fermion_kick(k + 1 < p->n_steps ? 2.0 * lam * e : lam * e));
    }
    return RHMC_OK;
  }
};

rhmc_status_t check_md(const rhmc_rational_t *md, const rhmc_md_params_t *p, const void *Phi, int n_pf) {
  if (!p || p->n_steps < 1 || p->n_gauge < 1 || !(p->tau >= 0.0) || !std::isfinite(p->lambda) ||
      !std::isfinite(p->beta)) {
    set_error("md parameters: need n_steps >= 1, n_gauge >= 1, finite tau >= 0, lambda and beta");
    return RHMC_ERR_INVALID_ARG;
  }
  if (Phi && n_pf > 0) {
    if (n_pf > RHMC_MAX_NRHS || !md || !md->alpha || !md->beta || md->n_shifts < 1 ||
        md->n_shifts > RHMC_MAX_SHIFTS) {
      set_error("md rational: need 1 <= n_shifts <= %d, alpha and beta, and n_pf <= %d", RHMC_MAX_SHIFTS,
                RHMC_MAX_NRHS);
      return RHMC_ERR_INVALID_ARG;
    }
    if (p->precision_md != RHMC_FP64 && p->precision_md != RHMC_MIXED_FP32) {
      set_error("md precision must be RHMC_FP64 or RHMC_MIXED_FP32");
      return RHMC_ERR_INVALID_ARG;
    }
  }
  return RHMC_OK;
}
}  // namespace

}  // namespace rhmc

using namespace rhmc;

namespace {
struct Guard {
  int prev = -1;
  explicit Guard(int dev) {
    cudaGetDevice(&prev);
    if (prev != dev) cudaSetDevice(dev);
  }
  ~Guard() {
    int cur = -1;
    cudaGetDevice(&cur);
    if (prev >= 0 && cur != prev) cudaSetDevice(prev);
  }
};
}  // namespace

#define RHMC_LATTICE(c, L)                                                    \
  Lat L;                                                                       \
  if (!(c)) {                                                                  \
    set_error("null context");                                                 \
    return RHMC_ERR_INVALID_ARG;                                               \
  }                                                                            \
  RHMC_TRY(lattice(c, &L));                                                    \
  Guard dg_(L.device);                                                         \
  CtxTuneScope ts_(c)

extern "C" {

rhmc_status_t rhmc_gauge_action(rhmc_ctx_t *c, const void *U, double beta, double *S_out, rhmc_stream_t sv) {
  RHMC_LATTICE(c, L);
  if (!U || !S_out) {
    set_error("rhmc_gauge_action: null U or S_out");
    return RHMC_ERR_INVALID_ARG;
  }
  return gauge_action(c, L.g, (const double2 *)U, beta, S_out, (cudaStream_t)sv);
}

rhmc_status_t rhmc_kinetic_energy(rhmc_ctx_t *c, const void *P, double *K_out, rhmc_stream_t sv) {
  RHMC_LATTICE(c, L);
  if (!P || !K_out) {
    set_error("rhmc_kinetic_energy: null P or K_out");
    return RHMC_ERR_INVALID_ARG;
  }
  return kinetic_energy(c, L.g, (const double2 *)P, K_out, (cudaStream_t)sv);
}

rhmc_status_t rhmc_momenta_from_normals(rhmc_ctx_t *c, const double *p, void *P, rhmc_stream_t sv) {
  RHMC_LATTICE(c, L);
  if (!p || !P) {
    set_error("rhmc_momenta_from_normals: null p or P");
    return RHMC_ERR_INVALID_ARG;
  }
  return momenta_from_normals(L.g, p, (double2 *)P, (cudaStream_t)sv);
}

rhmc_status_t rhmc_gauge_momentum(rhmc_ctx_t *c, const void *U, void *P, double beta, double eps, rhmc_stream_t sv) {
  RHMC_LATTICE(c, L);
  if (!U || !P) {
    set_error("rhmc_gauge_momentum: null U or P");
    return RHMC_ERR_INVALID_ARG;
  }
  return gauge_momentum(c, L.g, (const double2 *)U, (double2 *)P, beta, eps, (cudaStream_t)sv);
}

rhmc_status_t rhmc_momentum_update(rhmc_ctx_t *c, const void *U, const void *G, void *P, double eps,
                                   rhmc_stream_t sv) {
  RHMC_LATTICE(c, L);
  if (!U || !G || !P) {
    set_error("rhmc_momentum_update: null U, G or P");
    return RHMC_ERR_INVALID_ARG;
  }
  return momentum_update(L.g, (const double2 *)U, (const double2 *)G, (double2 *)P, eps, (cudaStream_t)sv);
}

rhmc_status_t rhmc_link_update(rhmc_ctx_t *c, void *U, const void *P, double eps, rhmc_stream_t sv) {
  RHMC_LATTICE(c, L);
  if (!U || !P) {
    set_error("rhmc_link_update: null U or P");
    return RHMC_ERR_INVALID_ARG;
  }
  return link_update(L.g, (double2 *)U, (const double2 *)P, eps, (cudaStream_t)sv);
}

rhmc_status_t rhmc_md_evolve(rhmc_ctx_t *c, void *U, void *P, const void *Phi, int n_pf, const rhmc_rational_t *md,
                             const rhmc_md_params_t *p, rhmc_md_info_t *info, rhmc_stream_t sv) {
  RHMC_LATTICE(c, L);
  if (!U || !P || (Phi && n_pf < 1)) {
    set_error("rhmc_md_evolve: null U or P, or pseudofermions with n_pf < 1");
    return RHMC_ERR_INVALID_ARG;
  }
  RHMC_TRY(check_md(md, p, Phi, n_pf));
  rhmc_md_info_t local{};
  if (!info) info = &local;
  *info = rhmc_md_info_t{};
  void *buf = nullptr;
  if (Phi) RHMC_TRY(ctx_md_buffer(c, (size_t)L.g.V * 4 * kLinkBytes, &buf));
  Md m{c, L.g, (double2 *)U, (double2 *)P, (double2 *)buf, Phi, Phi ? n_pf : 0, md, p, info, (cudaStream_t)sv};
  RHMC_TRY(m.run());
  // the context's staged links follow U
  return rhmc_set_gauge(c, U, sv);
}

rhmc_status_t rhmc_hmc_trajectory(rhmc_ctx_t *c, void *U, const double *pn, const void *eta, int n_pf,
                                  const rhmc_rational_t *hb, const rhmc_rational_t *md, const rhmc_rational_t *act,
                                  const rhmc_md_params_t *p, double tol_action, double u_accept, void *Phi_out,
                                  rhmc_hmc_info_t *info, rhmc_stream_t sv) {
  RHMC_LATTICE(c, L);
  const bool ferm = eta != nullptr;
  if (!U || !pn || (ferm && (n_pf < 1 || n_pf > RHMC_MAX_NRHS)) || !(tol_action > 0.0)) {
    set_error("rhmc_hmc_trajectory: null U or p, n_pf out of [1, %d] with eta, or tol_action <= 0", RHMC_MAX_NRHS);
    return RHMC_ERR_INVALID_ARG;
  }
  for (const rhmc_rational_t *r : {hb, act})
    if (ferm && (!r || !r->alpha || !r->beta || r->n_shifts < 1 || r->n_shifts > RHMC_MAX_SHIFTS)) {
      set_error("rhmc_hmc_trajectory: heatbath and action rationals need 1 <= n_shifts <= %d", RHMC_MAX_SHIFTS);
      return RHMC_ERR_INVALID_ARG;
    }
  RHMC_TRY(check_md(md, p, ferm ? eta : nullptr, n_pf));
  cudaStream_t s = (cudaStream_t)sv;
  rhmc_hmc_info_t local{};
  if (!info) info = &local;
  *info = rhmc_hmc_info_t{};

  // buffer: momenta | trial links | force | pseudofermions
  const size_t fld = (size_t)L.g.V * 4 * kLinkBytes;
  const size_t pf = ferm ? (size_t)L.g.Vh * 3 * n_pf * sizeof(double2) : 0;
  void *buf = nullptr;
  RHMC_TRY(ctx_md_buffer(c, 3 * fld + pf, &buf));
  double2 *P = (double2 *)buf;
  double2 *U1 = (double2 *)((char *)buf + fld);
  double2 *G = (double2 *)((char *)buf + 2 * fld);
  double2 *Phi = ferm ? (double2 *)((char *)buf + 3 * fld) : nullptr;

  RHMC_TRY(momenta_from_normals(L.g, pn, P, s));
  RHMC_TRY(rhmc_set_gauge(c, U, sv));
  auto fermion_action = [&](double *Sf) -> rhmc_status_t {
    *Sf = 0.0;
    if (!ferm) return RHMC_OK;
    return rhmc_force(c, Phi, n_pf, act->alpha0, act->alpha, act->beta, act->n_shifts, tol_action, 0, RHMC_FP64,
                      nullptr, nullptr, Sf, nullptr, nullptr, sv);
  };
  if (ferm) {
    RHMC_TRY(rhmc_rational_solve(c, eta, n_pf, hb->alpha0, hb->alpha, hb->beta, hb->n_shifts, tol_action, 0, Phi,
                                 nullptr, nullptr, sv));
    if (Phi_out) RHMC_CUDA_TRY(cudaMemcpyAsync(Phi_out, Phi, pf, cudaMemcpyDeviceToDevice, s));
  }
  RHMC_TRY(kinetic_energy(c, L.g, P, &info->K[0], s));
  RHMC_TRY(gauge_action(c, L.g, (const double2 *)U, p->beta, &info->S_g[0], s));
  RHMC_TRY(fermion_action(&info->S_f[0]));
  info->H_old = info->K[0] + info->S_g[0] + info->S_f[0];

  RHMC_CUDA_TRY(cudaMemcpyAsync(U1, U, fld, cudaMemcpyDeviceToDevice, s));
  Md m{c, L.g, U1, P, G, Phi, ferm ? n_pf : 0, md, p, &info->md, s};
  RHMC_TRY(m.run());

  RHMC_TRY(rhmc_set_gauge(c, U1, sv));
  RHMC_TRY(kinetic_energy(c, L.g, P, &info->K[1], s));
  RHMC_TRY(gauge_action(c, L.g, U1, p->beta, &info->S_g[1], s));
  RHMC_TRY(fermion_action(&info->S_f[1]));
  info->H_new = info->K[1] + info->S_g[1] + info->S_f[1];
  info->dH = info->H_new - info->H_old;
  info->accepted = (info->dH <= 0.0 || u_accept < std::exp(-info->dH)) ? 1 : 0;
  if (info->accepted) {
    RHMC_CUDA_TRY(cudaMemcpyAsync(U, U1, fld, cudaMemcpyDeviceToDevice, s));
    RHMC_CUDA_TRY(cudaStreamSynchronize(s));
  } else {
    RHMC_TRY(rhmc_set_gauge(c, U, sv));
  }
  return RHMC_OK;
}

}  // extern "C"
