// Internal launch wrappers (host functions enqueueing kernels on a stream).
#pragma once

#include "common.cuh"

// Instantiate a launch for the runtime width n = 1..16.
#define RHMC_DISPATCH_N(n, MACRO) \
  switch (n) {                    \
    case 1: MACRO(1); break;      \
    case 2: MACRO(2); break;      \
    case 3: MACRO(3); break;      \
    case 4: MACRO(4); break;      \
    case 5: MACRO(5); break;      \
    case 6: MACRO(6); break;      \
    case 7: MACRO(7); break;      \
    case 8: MACRO(8); break;      \
    case 9: MACRO(9); break;      \
    case 10: MACRO(10); break;    \
    case 11: MACRO(11); break;    \
    case 12: MACRO(12); break;    \
    case 13: MACRO(13); break;    \
    case 14: MACRO(14); break;    \
    case 15: MACRO(15); break;    \
    case 16: MACRO(16); break;    \
    default: return RHMC_ERR_INVALID_ARG; \
  }

namespace rhmc {

constexpr int kMaxN = RHMC_MAX_NRHS;
constexpr int kMaxS = RHMC_MAX_SHIFTS;

// Device-resident state of the SBCGrQ coefficient recursion (FP64).  Matrices
// are n x n row-major in the first n*n entries.  Slot k % kSlots holds
// iteration k's alpha, Gram1 (= alpha^-1), rho and delta: the shifted
// coefficient step of iteration k reads slots k and k-1 while the base step of
// iteration k+1 already writes slot k+1 on another stream.
constexpr int kSlots = 3;
struct SolverState {
  double2 alpha[kSlots][kMaxN * kMaxN];
  double2 G1[kSlots][kMaxN * kMaxN];
  double2 rho[kSlots][kMaxN * kMaxN];
  double2 delta[kSlots][kMaxN * kMaxN];
  double2 m2_s[kMaxS][kMaxN * kMaxN];   // beta^(s)_k rho_k^dagger of the last update of shift s
  double2 alpha_s[kMaxS][kMaxN * kMaxN];
  double sigma[kMaxS];        // shifts, ascending
  double d0[kMaxN];           // ||B e_j||
  double inv_d0[kMaxN];       // 1 / ||B e_j||
  double w1[kMaxS];           // weight of shift s's solution update (accumulating solves), 1 otherwise
  double res[kMaxS][kMaxN];   // recursive relative residual per shift and column (s = 0: base)
  int active[kMaxS];          // shift still being updated
  int upd[kMaxS];             // shift updated in the current iteration
  int last_k[kMaxS];          // last iteration that updated shift s (stored-basis mode)
  int kabs[kSlots];           // absolute iteration number of slot k % kSlots (graph replays reuse k's slot)
  int breakdown;              // nonzero: which coefficient step failed
  int device_timeout;         // a bounded device-side wait expired
  int done;                   // the base residuals are below stop_tol: later iterations change nothing
  int nit;                    // iterations run (device count; up to the one that set done)
  double stop_tol;            // > 0: stop on the device once every base residual is below (single shift, mixed)
  double a0;                  // 4 m^2 + sigma_0 (the mixed solve's operator reads it here)
};

// dslash.cu
rhmc_status_t stage_links(const Geom &g, const double2 *U, int bc_t, double2 *l64[2], float2 *l32[2],
                          cudaStream_t s);
// links12: optional 12-real copy of `links` (FP32 single-field hops use it), bc_t
// its boundary condition (signs of the rebuilt third rows); st (optional, all-directions
// kernel): a is read from st->a0 and nothing is done once st->done is set
template <typename T>
rhmc_status_t hop(const Geom &g, int par, const C<T> *links, const C<T> *in, C<T> *out, const C<T> *self, double a,
                  int n, int nbatch, long bstride, cudaStream_t s, const C<T> *links12 = nullptr, int bc_t = -1,
                  const SolverState *st = nullptr);
rhmc_status_t stage_links12(const Geom &g, int bc_t, float2 *const l32[2], float2 *l12[2], bool *ok, cudaStream_t s);

// FP64-accurate operator on the integer units (fx.cuh): integer link records (int4 per
// complex), the exponent of each site's largest entry, and the FP64 records
struct FxLinks {
  const int4 *rec = nullptr;
  const int *exp = nullptr;
  const double2 *l64 = nullptr;
};
// a field in integer form: int4 per complex [sites][3][n], exponent per (site, column)
struct FxField {
  int4 *v = nullptr;
  int *e = nullptr;
};
rhmc_status_t stage_links_fx(const Geom &g, const double2 *l64, int4 *lfx, int *lexp, cudaStream_t s);
// out = D in for an FP64 field, out in integer form (cat: profiler category); conv: an
// FP64-sized buffer and exponents for the converted input
rhmc_status_t hop_fx(const Geom &g, int par, const FxLinks &L, const double2 *in, FxField conv, FxField out, int n,
                     int cat, cudaStream_t s);
// the same with FP64 output (conv may be empty; the values and then the exponents take
// hop_fx_conv_bytes, 0 where it would not be used), and as double-float pairs
size_t hop_fx_conv_bytes(const Geom &g, int n);
rhmc_status_t hop_fx_to64(const Geom &g, int par, const FxLinks &L, const double2 *in, FxField conv, double2 *out,
                          int n, cudaStream_t s);
rhmc_status_t hop_fx_to_df(const Geom &g, int par, const FxLinks &L, const double2 *in, FxField conv, float4 *out,
                           int n, cudaStream_t s);
// out = a self - D in for an input in integer form, FP64 output
rhmc_status_t hop_fx_self(const Geom &g, int par, const FxLinks &L, FxField in, double2 *out, const double2 *self,
                          double a, int n, cudaStream_t s);
// R = B - (a X - D_eo tmp) (tmp = D_oe X), with the optional FP32 copy Rf and the nparts x n
// column partials of |R|^2 (part; scratch: hop_fx_parts x n doubles)
long hop_fx_parts(const Geom &g, int n);
rhmc_status_t resid_fx(const Geom &g, const FxLinks &L, FxField tmp, const double2 *X, double a, const double2 *B,
                       double2 *R, float2 *Rf, int n, double *scratch, double *part, int nparts, cudaStream_t s);
rhmc_status_t df_split(const double2 *in, float4 *out, long len, cudaStream_t s);

// blas.cu
constexpr int kGramCtas = 4 * 152;  // CTAs of the Gram kernel (its scratch holds kGramCtas * n * n partials)
// G = A^dagger B into out; with nparts and few CTAs their partials stay in scratch
// ([entry][part]) for the n x n kernel to sum: *nparts > 1, else 1
template <typename T>
rhmc_status_t gram(const C<T> *A, const C<T> *B, long rows, int n, double2 *scratch, double2 *out, cudaStream_t s,
                   const int *done = nullptr, int *nparts = nullptr);
template <typename TA, typename TY>
rhmc_status_t block_axpy(const C<TA> *A, const C<TY> *Cin, const C<TA> *M, C<TY> *Y, long rows, int n,
                         cudaStream_t s);
// Shifts [s_begin, s_end): X^(s) += P^(s) M1^(s), P^(s) = Q + P^(s) M2^(s).
// compute_q: first form Q = W rho^-1 (and store it); otherwise read Q.
template <typename T, typename TX>
rhmc_status_t update_all(const C<T> *W, C<T> *Q, C<T> *P, C<TX> *X, const C<T> *coef, const int *upd, int s_begin,
                         int s_end, int compute_q, long rows, int n, long fstride, cudaStream_t s, int acc = 0);
rhmc_status_t flush(double2 *X64, float2 *X32, long len, cudaStream_t s);

// update_tc.cu: shifted updates on the tensor cores (mixed path, n = 16)
// Y = C + A M (FP32, C may be null) with column-owner lanes and cp.async-staged row tiles
rhmc_status_t axpy_cols(const float2 *A, const float2 *C, const float2 *M, float2 *Y, long rows, int n,
                        cudaStream_t s);
// Y = C + A M fused with out = Y^dagger Y (n x n FP64, scratch: kGramCtas * n * n partials)
rhmc_status_t axpy_gram_cols(const float2 *A, const float2 *C, const float2 *M, float2 *Y, long rows, int n,
                             double2 *scratch, double2 *out, cudaStream_t s, const int *done = nullptr,
                             int *nparts = nullptr);
// The base step after rho_k in one pass: Q = W rho^-1, X^(0) += P^(0) M1, P^(0) = Q + P^(0) M2
// (coef: rho^-1, M1, M2), and Q into basis block *kdev when basis is given (capacity cap);
// nothing when *upd is 0
rhmc_status_t base_step(const float2 *W, float2 *Q, float2 *P, float2 *X, const float2 *coef, float2 *basis, int cap,
                        const int *kdev, const int *upd, long rows, int n, cudaStream_t s);
// FP32 shifted updates (Algorithm 1) with column-owner lanes and cp.async-staged row tiles
rhmc_status_t update_shifts_cols(const float2 *Q, float2 *P, float2 *X, const float2 *coef, const int *upd,
                                 int s_begin, int s_end, long rows, int n, long fstride, cudaStream_t s);
rhmc_status_t update_shifts_tc(const float2 *Q, float2 *P, float2 *X, const float2 *coef, const int *upd,
                               int s_begin, int s_end, long rows, long fstride, float *btiles, int *err,
                               cudaStream_t s);
template <typename TI, typename TO>
rhmc_status_t convert(const C<TI> *in, C<TO> *out, long len, cudaStream_t s);
rhmc_status_t sub(const double2 *a, const double2 *b, double2 *out, long len, cudaStream_t s);
rhmc_status_t add_inplace(double2 *a, const double2 *b, long len, cudaStream_t s);
template <typename T>
rhmc_status_t colnorm2(const C<T> *A, long rows, int n, double *partial, int nparts, cudaStream_t s);
rhmc_status_t redot(const double2 *A, const double2 *B, long len, double *partial, int nparts, cudaStream_t s);

// small.cu
template <typename T>
rhmc_status_t nxn_qr_init(const double2 *partial, int nparts, int n, int nshift, SolverState *st, C<T> *rinv,
                          cudaStream_t s);
template <typename T>
rhmc_status_t nxn_alpha(const double2 *partial, int nparts, int n, SolverState *st, int k, C<T> *mw, cudaStream_t s);
// small_df.cu: double-float forms of nxn_alpha / nxn_rho for the mixed solve ([entry][part] Gram partials)
rhmc_status_t nxn_alpha_dd(const double2 *gram, int nparts, int n, SolverState *st, int k, float2 *mw, cudaStream_t s);
rhmc_status_t nxn_rho_dd(const double2 *gram, int nparts, int n, SolverState *st, int k, float2 *coef, cudaStream_t s);
rhmc_status_t nxn_shifts_dd(int n, int nshift, SolverState *st, int k, float2 *coef, double tol_shift, int freeze,
                            double2 *hist, int cap, cudaStream_t s);
template <typename T>
rhmc_status_t nxn_rho(const double2 *partial, int nparts, int n, SolverState *st, int k, C<T> *coef, cudaStream_t s);
// hist (nullable, stored-basis mode): [cap][nshift][2][n*n] FP64, alpha^(s)_k and
// beta^(s)_k rho_k^dagger recorded at iteration k < cap
template <typename T>
rhmc_status_t nxn_shifts(int n, int nshift, SolverState *st, int k, C<T> *coef, double tol_shift, int freeze,
                         double2 *hist, int cap, cudaStream_t s);
// Stored-basis mode (basis.cu).  Buffers of the assembly: the block basis
// (rows x cap*n FP32 complex, row-major), the recorded per-iteration shift
// coefficients hist [cap][nshift][2][n*n] (alpha^(s)_k, beta^(s)_k rho_k^dagger),
// FP64 expansion coefficients cf [nshift-1][cap+1][n*n], the packed FP16 operand
// tiles of the tensor-core kernel (basis_pack_bytes), per-shift scales and per-tile
// K extents.
struct BasisBufs {
  float2 *basis = nullptr;
  double2 *hist = nullptr;
  double2 *cf = nullptr;
  unsigned char *bpack = nullptr;
  double *bscale = nullptr;  // [nshift]
  int *tile_nkt = nullptr;   // [nshift]
  int cap = 0;
};
size_t basis_pack_bytes(int n, int nshift, int cap);
// cf of basis_assemble (FP64 expansion coefficients of X^(s) or P^(s)) alone
rhmc_status_t basis_coef(const BasisBufs &bb, int n, int nshift, const SolverState *st, int K, int want_p,
                         cudaStream_t s);
// basis64.cu: the FP64 solve's stored basis, a device table of blocks [rows][n]; kdev: the device's iteration
// counter k.  W = Q_{k-1} + A M; Q_k = W rho^-1, X^(0) += P M1, P = Q_k + P M2.
rhmc_status_t axpy64(const double2 *A, double2 *const *basis, const int *kdev, const double2 *M, double2 *Y, long rows,
                     int n, cudaStream_t s);
rhmc_status_t base64(const double2 *W, double2 *const *basis, const int *kdev, double2 *P, double2 *X, const double2 *coef,
                     long rows, int n, cudaStream_t s);
// out_s = X^(s) (want_p = 0) or P^(s)_K (want_p = 1, active shifts) for s = 1 .. nshift - 1, at
// out + (s - 1) fstride; combine (want_p = 0): sum_s w_s X^(s) into out.  bb.hist, bb.cf (room
// for nshift sets of cap + 1 blocks) and bb.cap are used.
rhmc_status_t basis64_assemble(const BasisBufs &bb, double2 *const *basis, int n, int nshift, const SolverState *st,
                               long rows, int K, int want_p, int combine, double2 *out, long fstride, cudaStream_t s);
// want_p = 0: X^(s) = sum_{i < last_s} Q_i C_i for s = 1 .. nshift-1 (FP64, C_i = alpha_{i+1}
// + M2_{i+1} C_{i+1}; X^(s), s >= 1, is overwritten: it is zero before the one assembly of a
// solve); want_p = 1: P^(s) = sum_{i <= K} Q_i D_i (FP32, D_K = 1, D_i = M2_{i+1} D_{i+1}),
// active shifts only.  chunk_blocks > 0 (X only): FP32 partial sums over about that many
// blocks, added in FP64.  simt: CUDA-core kernel instead of tcgen05.  acc_kt: K tiles (of 64
// reals) per tensor-memory accumulation chunk (0: built-in).  err: device flag set when a
// bounded wait of the tensor-core kernel gave up.
rhmc_status_t basis_assemble(const BasisBufs &bb, int n, int nshift, const SolverState *st, long rows, int K,
                             int want_p, double2 *X, float2 *P, long fstride, int chunk_blocks, int simt, int acc_kt,
                             int *err, cudaStream_t s);
// Q (rows x n) into column block k of the basis (rows x cap*n, row-major)
rhmc_status_t basis_store(const float2 *Q, float2 *basis, long rows, int n, int cap, int k, cudaStream_t s);
// the same with the block index read from *kdev (an iteration counter in device memory)
rhmc_status_t basis_store_dev(const float2 *Q, float2 *basis, long rows, int n, int cap, const int *kdev,
                              cudaStream_t s);
template <typename T>
rhmc_status_t nxn_reliable(const double2 *partial, int nparts, int n, SolverState *st, int k, C<T> *rinv,
                           cudaStream_t s);

// force.cu
rhmc_status_t rational_combine(const double2 *Phi, double alpha0, const double *alpha_host, const double2 *X, int ns,
                               long len, double2 *Y, cudaStream_t s);
// the same from double-float fields (float4 per complex)
rhmc_status_t force_links_df(const Geom &g, const float4 *X, const float4 *Y, int n, int nshift, long fstride,
                             const double *alpha_dev, int bc_t, double2 *G, cudaStream_t s);
rhmc_status_t force_links(const Geom &g, const double2 *X, const double2 *Y, int n, int nshift, long fstride,
                          const double *alpha_dev, int bc_t, double2 *G, cudaStream_t s);
// F = TA(U G^dagger) per link (F may be null or alias G); partial[nparts]: per-CTA sums of |F|_F^2 / 4
rhmc_status_t force_lie(const Geom &g, const double2 *U, const double2 *G, double2 *F, double *partial, int nparts,
                        cudaStream_t s);

// api.cu: the calling thread uses ctx's launch settings (rhmc_ctx_tune_set) while
// an object of this type lives, as every entry point of api.cu does.
struct CtxTuneScope {
  const int *prev;
  explicit CtxTuneScope(const rhmc_ctx_t *c);
  ~CtxTuneScope();
};

// api.cu: read-only view of a context (device, geometry, mass, staged
// links of the two output parities); NO_GAUGE before rhmc_set_gauge.
rhmc_status_t ctx_geometry(const rhmc_ctx_t *ctx, int *device, Geom *g, double *mass, FxLinks *even, FxLinks *odd);

// api.cu: Y = (A + sigma) X in FP64 with caller scratch (tmp: FP64 field, exps: 2 Vh n)
rhmc_status_t apply_noalloc(const Geom &g, const FxLinks &even, const FxLinks &odd, double mass, const double2 *X,
                            double2 *Y, double2 *tmp, int *exps, int n, double sigma, cudaStream_t s);

// api.cu: device and geometry of a context (no gauge field needed), and its
// scratch array of per-CTA partial sums (allocated on first use)
rhmc_status_t ctx_lattice(const rhmc_ctx_t *ctx, int *device, Geom *g);
rhmc_status_t ctx_partials(rhmc_ctx_t *ctx, double **parts, int *nparts);
// api.cu: the context's molecular-dynamics buffer, at least `bytes` long (kept
// across calls, reallocated when too small)
rhmc_status_t ctx_md_buffer(rhmc_ctx_t *ctx, size_t bytes, void **buf);

// api.cu: the context's buffer for one set of links in integer form (4 V x 9 int4, then 4 V
// flags; allocated on first use).  begin makes stream s wait for the buffer's last user and
// gives nullptr where there is no memory or s is being captured; end marks s's use of it.
int4 *ctx_links_fx_begin(rhmc_ctx_t *c, cudaStream_t s);
rhmc_status_t ctx_links_fx_end(rhmc_ctx_t *c, cudaStream_t s);

// scg.cu (per-vector FP64 multishift CG baseline)
struct ScgState;

}  // namespace rhmc
