// BiCGStab's scalar recurrence: from the block partials of a system's dots to
// its alpha, omega, rho, beta and status, by a kernel of its own or, where the
// vectors are short (fin_fused), by the last block of the kernel that wrote the
// partials: 4.5 us more in that kernel instead of 7.2 us and a launch (4^4).
// Every block then waits for its stores before it arrives, which costs kernels
// with many blocks more than the launch (16^4, 10 systems: 364 ms a solve
// against 346; 16^3 x 32 in FP16 83 against 66).  The partials are summed in
// block order either way: results do not depend on which block comes last.
#pragma once

#include "cplx.cuh"
#include "kernels.cuh"

namespace wd {

// FIN_ALPHA, FIN_OMEGA or FIN_RHO of system r, status ST_ACTIVE, by a block of
// 128 threads or more.  An FP64 division, square root or hypot is a chain
// of ten or more FP64 instructions of 64 clocks each, so independent ones go to
// different warps.
static __device__ __noinline__ void fin_system(int kind, const double *partial, int nb, BicgScalars *sc,
                                               int *status, double *hist, int hist_len, int r) {
  __shared__ double sum[3];
  __shared__ double2 quot[2];
  __shared__ double root[2];
  BicgScalars &S = sc[r];
  double v[3] = {0.0, 0.0, 0.0};
  const double *src = partial + (long long)r * nb * 3;
#pragma unroll 4
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
#pragma unroll
    for (int q = 0; q < 3; ++q) v[q] += __ldcg(src + 3 * b + q);
  }
  block_sum<3>(v);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int q = 0; q < 3; ++q) sum[q] = v[q];
  }
  __syncthreads();
  const double2 d = make_double2(sum[0], sum[1]);
  const double n2 = sum[2];
  const int role = threadIdx.x % 32 == 0 ? threadIdx.x / 32 : 4;
  if (role == 0) {
    if (kind == FIN_ALPHA) quot[0] = cdiv(S.rho, d);
    else if (kind == FIN_OMEGA) quot[0].x = n2 == 0.0 ? 0.0 : d.x / n2;
    else quot[0] = cdiv(d, S.rho);   // rho / rho_old
  } else if (role == 1) {
    if (kind == FIN_OMEGA) quot[0].y = n2 == 0.0 ? 0.0 : d.y / n2;
    else root[0] = sqrt(n2);
  } else if (role == 2 && kind != FIN_OMEGA) {
    root[1] = hypot(d.x, d.y);
  } else if (role == 3 && kind == FIN_RHO) {
    quot[1] = cdiv(S.alpha, S.omega);
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  if (kind == FIN_ALPHA) {  // <r_hat, v>, ||v||^2
    S.mvp += 1;
    if (root[1] <= 1e-30 * S.rhat_norm * root[0]) {
      status[r] = ST_BREAKDOWN;
      return;
    }
    S.alpha = quot[0];
  } else if (kind == FIN_OMEGA) {  // <t, s>, ||t||^2
    // t = A s = 0 means s = 0: omega = 0, x += alpha p finishes
    if (n2 != 0.0) S.mvp += 1;
    S.omega = quot[0];
  } else {  // FIN_RHO: <r_hat, r>, ||r||^2
    const double rnorm = root[0], rel = rnorm / S.bnorm;
    const double2 beta = cmul(quot[0], quot[1]);
    S.beta = beta;
    S.mbo = cneg(cmul(beta, S.omega));
    S.rho_old = S.rho;
    S.rho = d;
    S.rnorm = rnorm;
    S.iters += 1;
    if (hist != nullptr && S.iters <= hist_len)
      hist[(long long)r * hist_len + S.iters - 1] = rel;
    if (rel <= S.tol)
      status[r] = ST_RECURSIVE;
    else if (S.iters >= S.max_iter)
      status[r] = ST_MAXITER;
    else if (root[1] <= 1e-30 * S.rhat_norm * rnorm)
      status[r] = ST_BREAKDOWN;
  }
}

// Called by every block of system r's launch after it wrote its partial
// (f.nb blocks): the last one to arrive finishes the scalar step.  Every block
// has read the system's status and scalars by then.  f.count == nullptr: none.
__device__ __forceinline__ void fin_last_block(const FinArgs &f, const double *partial, int r) {
  if (f.count == nullptr) return;
  __shared__ int last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();   // the block's partial (ordered by the barrier) before its arrival
    last = atomicAdd(f.count + r, 1u) == (unsigned)f.nb - 1u;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x == 0) f.count[r] = 0;
  fin_system(f.kind, partial, f.nb, f.sc, f.status, f.hist, f.hist_len, r);
}

}  // namespace wd
