// Kernel-level declarations shared by the CUDA translation units.
#pragma once

#include <cuda_runtime.h>

#include "wd_internal.h"

namespace wd {

struct LatticeGeom {
  int L[4];
  long long V;
  // Division by L[0], L[1], L[2] of site indices below 2^31 as a multiply
  // and a shift (Granlund and Montgomery, "Division by invariant integers
  // using multiplication", 1994): q = (n * dm) >> dsh with dsh = 31 + l,
  // l = ceil(log2 d), dm = floor(2^dsh / d) + 1, exact for n < 2^31.
  unsigned long long dm[3];
  int dsh[3];
  int split;   // all extents even: the fixed-point links are stored parity by parity
};

enum { EPI_NONE = 0, EPI_DOT = 1, EPI_TSTT = 2 };

// Per-system solver status.  Kernels take a bit mask of the statuses they
// act on and skip every other system.
enum SysStatus {
  ST_ACTIVE = 0,       // iterating
  ST_RECURSIVE = 1,    // recursive residual below tol: check the true one
  ST_BREAKDOWN = 2,    // final
  ST_MAXITER = 3,      // final
  ST_DONE = 4,         // true residual below tol: final
  ST_FAILED = 5,       // true residual above tol, restarts used up: final
  ST_RESTART = 6,      // transient: restart from the true residual
  ST_IDLE = 7          // not part of this phase
};
constexpr unsigned M_ACTIVE = 1u << ST_ACTIVE;
constexpr unsigned M_RECURSIVE = 1u << ST_RECURSIVE;
constexpr unsigned M_RESTART = 1u << ST_RESTART;
constexpr unsigned M_ALL = 0xffffffffu;

// BiCGStab scalars of one system, device resident.
struct BicgScalars {
  double2 rho, rho_old, alpha, omega;
  double2 beta, mbo;   // of the next p = r + beta p + mbo v: (rho / rho_old)(alpha / omega), -beta omega
  double bnorm, rhat_norm, rnorm, true_rel, tol;
  int iters, max_iter, restarts, max_restarts;
  int shadows;   // restarts with a new shadow vector (bicg_fin.cuh)
  long long mvp, mvp_extra;
  // mixed solver only: tol is the target of the low-precision recursion;
  // tol_outer the FP64 true-residual target; delta > 0 selects restarted
  // refinement (inner target delta x the residual at the last restart)
  double tol_outer, delta;
};

// A scalar step of BiCGStab to be done by the last block of the launch that
// writes its nb partials a system (bicg_fin.cuh): kind FIN_ALPHA, FIN_OMEGA or
// FIN_RHO; count: a zero a system; count == nullptr: no step.
struct FinArgs {
  int kind, nb;
  BicgScalars *sc;
  int *status;
  double *hist;
  int hist_len;
  unsigned *count;
};

LatticeGeom geom_of(const wd_context *h);

// Fixed-point spinors (fx.cuh): v [rhs][tile of 32 sites][12][32], e [rhs][sites].
struct FxVec {
  int4 *v;
  int *e;
};
constexpr int WILSON_SITES = 64;   // per block of the FP64 products, in fixed point and in FP64
// blocks (partials a system) of a product of nrhs systems, and whether it reads `pre`
int wilson_blocks(const wd_context *h, int nrhs);
bool wilson_takes_encoded(const wd_context *h, int nrhs);
cudaError_t fx_links_create(wd_context *h);
void fx_links_release(wd_context *h);   // waits for the device
// Whether s records a graph.  Products then take no scratch, hence the FP64
// kernels above the few-site size: a graph with allocation nodes could be
// neither instantiated twice nor cloned.
bool being_captured(cudaStream_t s);
// Encode nrhs vectors of `sites` sites (systems in mask).
cudaError_t launch_fx_encode(const double2 *in, FxVec f, long long sites, int nrhs,
                             const int *status, unsigned mask, cudaStream_t s);

// Wilson apply with an optional fused reduction epilogue; blocks of systems
// whose status is not in `mask` do nothing (status == nullptr: all act).
// pre: `in` already in fixed point (used when the handle has such links).
// fin: the scalar step on the epilogue's partials, nrhs systems.
cudaError_t launch_wilson_f64_epi(const wd_context *h, const double2 *in, double2 *out,
                                  int nrhs, int dagger, int epi, const double2 *aux,
                                  double *partial, const int *status, cudaStream_t s,
                                  unsigned mask = M_ACTIVE, const FxVec *pre = nullptr,
                                  const FinArgs *fin = nullptr);

// ----------------------------------------------------------------- BLAS1
// Number of blocks (per system) every streaming kernel uses; fixed so that
// the reduction order, and hence every result, is reproducible.
int stream_blocks(long long n);

// BiCGStab updates of the active systems in fixed point (fx_stream.cu); n a
// multiple of 12.  fx (v may be nullptr): the result site by site for the
// operator.  update_xr writes fxs_blocks(n, nrhs) partials (<rhat, r>, ||r||^2) a system.
int fxs_blocks(long long n, int nrhs);
// Whether the scalar steps of nrhs systems go to the last block of the kernels
// that form their dots.
bool fin_fused(long long n, int nrhs);
cudaError_t launch_bicg_update_p(double2 *p, const double2 *r, const double2 *v, FxVec fx,
                                 const BicgScalars *sc, const int *status, long long n,
                                 int nrhs, cudaStream_t s);
cudaError_t launch_bicg_update_s(double2 *sv, const double2 *r, const double2 *v, FxVec fx,
                                 const BicgScalars *sc, const int *status, long long n,
                                 int nrhs, cudaStream_t s);
cudaError_t launch_bicg_update_xr(double2 *x, double2 *r, const double2 *p, const double2 *sv,
                                  const double2 *t, const double2 *rhat, const BicgScalars *sc,
                                  const int *status, double *partial, long long n, int nrhs,
                                  const FinArgs &fin, cudaStream_t s);
// out = a - b, partial <- ||out||^2 ; systems in mask only
cudaError_t launch_sub_norm(double2 *out, const double2 *a, const double2 *b, const int *status,
                            unsigned mask, double *partial, long long n, int nrhs,
                            cudaStream_t s);
// partial <- ||a||^2 (and ||b||^2 when b != nullptr), all systems
cudaError_t launch_norms(const double2 *a, const double2 *b, double *partial, long long n,
                         int nrhs, cudaStream_t s);
// for systems in mask: rhat = r, p = 0, v = 0
cudaError_t launch_bicg_restart_vectors(double2 *rhat, const double2 *r, double2 *p,
                                        double2 *v, const int *status, unsigned mask,
                                        long long n, int nrhs, cudaStream_t s);

// Scalar finalizers (one block per system): reduce nb block partials of NQ
// doubles in a fixed order, then update the scalars and status.
enum FinKind { FIN_INIT, FIN_ALPHA, FIN_OMEGA, FIN_RHO, FIN_TRUE, FIN_ACTIVATE };
cudaError_t launch_bicg_finalize(int kind, const double *partial, int nb, BicgScalars *sc,
                                 int *status, double *hist, int hist_len, int nrhs,
                                 cudaStream_t s);

// ----------------------------------------------------------------- tall-skinny
// C[j][r] = sum_i conj(V[j][i]) * (g5 ? gamma5 W[r] : W[r])[i],  j < k, r < nrhs.
// launch_ts_dot writes ts_dot_blocks(n, k, nrhs) tiles of block partials to
// `partial` (k*nrhs complex per ... tile layout private to blas.cu, at most
// TS_MAX_BLOCKS * 16 complex); launch_ts_dot_finalize, given the same
// (n, k, nrhs), sums them in block order into C[j*ldc + r] and, when
// C2 != nullptr, also adds them to C2[j*ldc2 + r].
constexpr int TS_MAX_BLOCKS = 608;  // blocks of one ts_dot launch, all tiles
int ts_dot_blocks(long long n, int k, int nrhs);
inline size_t ts_dot_partial_count(long long n, int k, int nrhs) {
  return (size_t)ts_dot_blocks(n, k, nrhs) * 16;  // JT*RT = 16 for every tile shape
}
cudaError_t launch_ts_dot(const double2 *V, int k, const double2 *W, int nrhs, int g5,
                          long long n, double2 *partial, const int *status,
                          cudaStream_t s);
cudaError_t launch_ts_dot_finalize(const double2 *partial, long long n, int k, int nrhs,
                                   double2 *C, int ldc, double2 *C2, int ldc2,
                                   const int *status, cudaStream_t s);
// the same sum of partials laid out [(gy rows, gx blocks)][JT x RT]
cudaError_t launch_ts_dot_finalize_grid(const double2 *partial, int gx, int gy, int JT, int RT, int k,
                                        int nrhs, double2 *C, int ldc, double2 *C2, int ldc2,
                                        const int *status, cudaStream_t s);
// OUT[c][i] = (beta_one ? IN[c][i] : 0) + sign * sum_j V[j][i] Y[j*ldy + c],
// c < ncol, kv <= 128.  OUT may alias IN (in-place update) but not V.
cudaError_t launch_ts_update(const double2 *V, int kv, const double2 *Y, int ldy, int ncol,
                             const double2 *IN, double2 *OUT, int beta_one, double sign,
                             long long n, const int *status, cudaStream_t s);

// The same product on the tensor cores (exact-split BF16 emulation to FP64
// accuracy, tc_gemm.cu): kv <= 88, any ncol; OUT may alias IN but not V.
// scratch: ts_update_tc_scratch_bytes(kv, ncol, n) device bytes; *err (device)
// is set to 1 if a wait of the kernel gave up (never in normal operation).
bool ts_update_tc_supported(int kv, int ncol);
size_t ts_update_tc_scratch_bytes(int kv, int ncol, long long n);
cudaError_t launch_ts_update_tc(const double2 *V, int kv, const double2 *Y, int ldy, int ncol,
                                const double2 *IN, double2 *OUT, int beta_one, double sign,
                                long long n, void *scratch, int *err, cudaStream_t s);

// ----------------------------------------------------------------- Arnoldi helpers
// partial -> ||w||^2 reduced; H[(j+1)*ldh + j] = ||w||; v = w / ||w||;
// lucky breakdown when ||w|| <= lucky * ||w0|| sets *status = 1 and m_eff.
cudaError_t launch_arnoldi_normalize_finalize(const double *partial_w, int nb,
                                              const double *partial_w0, int nb0,
                                              double2 *H, int ldh, int j, double lucky,
                                              int *status, int *m_eff, cudaStream_t s);
// *dst = sqrt(sum_i partial[i*stride]) for i < nb (deterministic order)
cudaError_t launch_norm_finalize(const double *partial, int nb, int stride, double2 *dst,
                                 cudaStream_t s);
// ----------------------------------------------------------------- Gram-Schmidt in fixed point (fx_basis.cu)
// Basis vectors of n entries (n even) in fixed point: planes hi, lo [vector][n]
// and exponents ex [vector][fxb_chunks(n)].
struct FxBasis {
  int2 *hi, *lo;
  int *ex;
};
long long fxb_chunks(long long n);
// `count` vectors from w, the first into slot j of b: v = w / Re(H[idx]) (H nullptr: v = w);
// v (may be w, or nullptr) gets the FP64 values, fx (one vector; fx.v may be
// nullptr) the site-wise form of the operator.  Nothing when *status != 0.
cudaError_t launch_fxb_encode(const double2 *w, const double2 *H, int idx, double2 *v, FxBasis b,
                              long long j, int count, FxVec fx, long long n, const int *status,
                              cudaStream_t s);
// C[j ldc] = <V_j, w> (g5: <V_j, gamma5 w>), j < k, and C2[j ldc2] += it when C2 != nullptr.
// partial: fxb_dot_partials(n, k) complex numbers.  V: the FP64 vectors.
size_t fxb_dot_partials(long long n, int k);
cudaError_t launch_fxb_dot(FxBasis b, const double2 *V, int k, const double2 *w, int g5, long long n,
                           double2 *partial, double2 *C, int ldc, double2 *C2, int ldc2,
                           const int *status, cudaStream_t s);
// w -= sum_j V_j h[j ldh] (add: w +=), k <= 128
cudaError_t launch_fxb_update(FxBasis b, const double2 *V, int k, const double2 *h, int ldh, int add,
                              double2 *w, long long n, const int *status, cudaStream_t s);
// w -= V h for the second classical Gram-Schmidt pass: FP32 products when
// ||h||^2 <= 1e-20 (||w0||^2 - ||hsum||^2) (part_w: Wilson-kernel partials,
// [3 b + 2] = block b's share of ||w0||^2; hsum: column of both passes'
// coefficients, stride ldh), else FP64.  part_n[2 c] = chunk c's share of
// ||w||^2 afterwards.
cudaError_t launch_fxb_correction(FxBasis b, const double2 *V, int k, const double2 *h,
                                  const double2 *hsum, int ldh, const double *part_w, int nbw,
                                  double2 *w, long long n, double *part_n, const int *status,
                                  cudaStream_t s);

// ----------------------------------------------------------------- small dense (1 CTA)
// LU with partial pivoting of a k x k matrix (row-major), in place; piv[k].
// info[0] = 0 ok, 1 singular; info[1] bits of an estimate of cond (double).
cudaError_t launch_lu_factor(double2 *A, int k, int *piv, double *info, cudaStream_t s);
// Solve A Y = C for nrhs columns (C row-major k x nrhs, overwritten by Y).
cudaError_t launch_lu_solve(const double2 *LU, const int *piv, int k, double2 *C, int nrhs,
                            cudaStream_t s);

struct CycleEndArgs {
  const double2 *H;    // (m+1) x m row-major Hbar_m
  const double2 *c;    // m+1
  int m, k;
  const int *m_eff;    // Arnoldi columns actually built (lucky breakdown)
  double2 *d;          // m: least-squares solution
  double2 *rho;        // m+1: c - Hbar d
  double *res;         // [0] ||rho||
  double2 *P;          // (m+1) x (k+1) row-major
  double2 *Hk;         // (k+1) x k row-major: P^dagger Hbar P_k
  double2 *ck;         // k+1: P^dagger rho
  double2 *theta;      // k harmonic Ritz values
  int *flags;          // [0] eig failure, [1] lucky, [2] FP32 estimates rejected (FP64 path)
  double2 *work;       // scratch >= 2*(m+1)*(m+1) + 2*m*m + 4*m + 2 complex
  long long *clk;      // nullptr, or 10 slots: SM clock at phase boundaries, QR sweeps, rotations
  int do_restart;
  int eig32;           // 1: FP32 estimates refined in FP64 first, 0: FP64 QR iteration only
};
cudaError_t launch_gmresdr_cycle_end(const CycleEndArgs &a, cudaStream_t s);
size_t gmresdr_cycle_end_smem(int m);

// ----------------------------------------------------------------- even-odd (evenodd.cu)
// B full -> Bhat (even half); be, bo: scratch half vectors (nrhs each)
cudaError_t launch_eo_prepare(wd_context *h, const double2 *B, double2 *Bhat, double2 *be,
                              double2 *bo, int nrhs, cudaStream_t s);
// B full, Xe even half -> X full
cudaError_t launch_eo_reconstruct(wd_context *h, const double2 *B, const double2 *Xe, double2 *X,
                                  double2 *be, double2 *bo, int nrhs, cudaStream_t s);

// ----------------------------------------------------------------- gradients (force.cu)
cudaError_t launch_link_force(const wd_context *h, const double2 *lam, const double2 *x, double *f,
                              cudaStream_t s);
// partial[b] (stream_blocks(n) of them) of Re sum conj(lam) (x + i mu g5 x - ax)
cudaError_t launch_dkappa(const double2 *lam, const double2 *x, const double2 *ax, double mu,
                          long long n, double *partial, cudaStream_t s);
cudaError_t launch_gamma5(const double2 *in, double2 *out, long long n, cudaStream_t s);

}  // namespace wd
