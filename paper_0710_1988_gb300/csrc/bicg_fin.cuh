// BiCGStab's scalar recurrence: from the block partials of a system's dots to
// its alpha, omega, rho, beta and status, by a kernel of its own or, where the
// vectors are short (fin_fused), by the last block of the kernel that wrote the
// partials: 4.5 us more in that kernel instead of 7.2 us and a launch (4^4).
// Every block then waits for its stores before it arrives, which costs kernels
// with many blocks more than the launch (16^4, 10 systems: 364 ms a solve
// against 346; 16^3 x 32 in FP16 83 against 66).  The partials are summed by
// their index either way: results do not depend on which block comes last.
// Sums in integers, the scalars loaded first: 13.9 -> 9 us for 4000 partials a
// system (20^3 x 32, 12 systems in FP32: 458 -> 437 ms a solve), 8.2 -> 7.0 us for
// 512; sums in FP64 keep one SM's pipe busy for 3.8 us of the former.
#pragma once

#include "cplx.cuh"
#include "fx.cuh"
#include "kernels.cuh"

namespace wd {

// Sums of three quantities over a warp, N <= 4 entries of each a lane, in all
// lanes: integers against each quantity's largest exponent field (fx.cuh), to
// 2^-56 of the largest entry, entries within 4 of it exactly.  A warp's FP64
// additions would take 76 clocks of its scheduler each, fifteen of them for
// the shuffles alone.
template <int N>
__device__ __forceinline__ void fin_warp_sum(const double (&x)[N][3], double (&sum)[3]) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    int e = 0;
    bool any = false;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      e = max(e, exp_bits(x[i][q]));
      any = any || (__double_as_longlong(x[i][q]) << 1) != 0;
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (e <= FX_EMAX && (e >= FX_EMIN || !__any_sync(0xffffffffu, any))) {
      e = max(e, FX_EMIN);   // zeros are shifted out, also where all entries are zero
      long long t = 0;
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const unsigned h = (unsigned)__double2hiint(x[i][q]);
        unsigned long long y = (unsigned long long)((h & 0xfffffu) | 0x100000u) << 32 |
                               (unsigned)__double2loint(x[i][q]);
        asm("shr.u64 %0, %1, %2;" : "=l"(y) : "l"(y << 3), "r"((unsigned)e - ((h >> 20) & 0x7ffu)));
        const long long m = (int)h >> 31;
        t += ((long long)((y + 1) >> 1) ^ m) - m;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      sum[q] = fx_scaled(t, e + 2);
    } else {   // infinities, NaN, magnitudes near the ends of the range
      double t = 0.0;
#pragma unroll
      for (int i = 0; i < N; ++i) t += x[i][q];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      sum[q] = t;
    }
  }
}

// The same over four of the nb partials of a system a lane: b, b + step, ...
__device__ __forceinline__ void fin_partials(const double *src, int b, int step, int nb, double (&sum)[3]) {
  double x[4][3];
#pragma unroll
  for (int i = 0; i < 4; ++i, b += step) {
#pragma unroll
    for (int q = 0; q < 3; ++q) x[i][q] = b < nb ? __ldcg(src + 3 * b + q) : 0.0;
  }
  fin_warp_sum(x, sum);
}

// The recurrence starts anew from r_hat = r, p = v = 0; rr = ||r||^2.
__device__ __forceinline__ void reset_recurrence(BicgScalars &S, double rr) {
  S.rho = make_double2(rr, 0.0);  // r_hat = r, so <r_hat, r> = ||r||^2
  S.rho_old = make_double2(1.0, 0.0);
  S.alpha = make_double2(1.0, 0.0);
  S.omega = make_double2(1.0, 0.0);
  S.beta = S.rho;
  S.mbo = cneg(S.rho);
  S.rhat_norm = sqrt(rr);
  S.rnorm = sqrt(rr);
}

// FIN_RHO with <r_hat, r> = 0 starts the recurrence anew from r this often.  It
// happens at the first step to sources on one site, whose r is orthogonal to them:
// A A b has no part at the site, as (1 - gamma)(1 + gamma) = 0.  In FP64 sums the
// rounding of alpha mostly hides it, with the more exact ones it shows.
constexpr int SHADOWS_MAX = 3;

// FIN_ALPHA, FIN_OMEGA or FIN_RHO of system r, status ST_ACTIVE, by a block of
// 128 threads or more.  What takes time is one chain: up to 128 partials are
// summed by each warp that needs them, without a barrier; the scalars are
// loaded before the partials, independent divisions and roots (ten or more
// FP64 instructions of 64 clocks each) go to different warps.
static __device__ __noinline__ void fin_system(int kind, const double *partial, int nb, BicgScalars *sc,
                                               int *status, double *hist, int hist_len, int r) {
  __shared__ double part[32][3];
  __shared__ double2 quot[2];
  __shared__ double root[2];
  BicgScalars &S = sc[r];
  const double2 rho = S.rho, alpha = S.alpha, omega = S.omega;
  const double bnorm = S.bnorm, rhat_norm = S.rhat_norm, tol = S.tol;
  const int iters = S.iters + 1, max_iter = S.max_iter;
  const long long mvp = S.mvp + 1;
  const int w = threadIdx.x / 32, lane = threadIdx.x % 32;
  const double *src = partial + (long long)r * nb * 3;
  double t[3];
  if (nb <= 128) {   // each of the four warps sums them all
    if (w >= 4) return;
    fin_partials(src, lane, 32, nb, t);
  } else {
    fin_partials(src, threadIdx.x, blockDim.x, nb, t);
    for (int b = 4 * blockDim.x; b < nb; b += 4 * blockDim.x) {
      double v[3];
      fin_partials(src, b + threadIdx.x, blockDim.x, nb, v);
#pragma unroll
      for (int q = 0; q < 3; ++q) t[q] += v[q];
    }
    if (lane < 3) part[w][lane] = lane == 0 ? t[0] : lane == 1 ? t[1] : t[2];
    __syncthreads();
    if (w >= 4) return;
    double x[1][3];
#pragma unroll
    for (int q = 0; q < 3; ++q) x[0][q] = lane < (int)blockDim.x / 32 ? part[lane][q] : 0.0;
    fin_warp_sum(x, t);
  }
  const double2 d = make_double2(t[0], t[1]);
  const double n2 = t[2];
  if (lane == 0) {
    if (w == 0) {
      if (kind == FIN_ALPHA) quot[0] = cdiv(rho, d);
      else if (kind == FIN_OMEGA) quot[0].x = n2 == 0.0 ? 0.0 : d.x / n2;
      else quot[0] = cdiv(d, rho);   // rho / rho_old
    } else if (w == 1) {
      if (kind == FIN_OMEGA) {
        quot[0].y = n2 == 0.0 ? 0.0 : d.y / n2;
      } else {
        const double n = sqrt(n2);
        root[0] = n;
        if (kind == FIN_RHO) root[1] = n / bnorm;
      }
    } else if (w == 3 && kind == FIN_RHO) {
      quot[1] = cdiv(alpha, omega);
    }
  }
  asm volatile("bar.sync 1, 128;" ::: "memory");   // the four warps
  if (threadIdx.x != 0) return;
  // |d| <= 1e-30 |r_hat| n, the square root only where the larger component says so
  const double limit = kind == FIN_OMEGA ? 0.0 : 1e-30 * rhat_norm * root[0];
  const bool vanishes = kind != FIN_OMEGA && !(fmax(fabs(d.x), fabs(d.y)) > limit) && hypot(d.x, d.y) <= limit;
  if (kind == FIN_ALPHA) {  // <r_hat, v>, ||v||^2
    S.mvp = mvp;
    if (vanishes) {
      status[r] = ST_BREAKDOWN;
      return;
    }
    S.alpha = quot[0];
  } else if (kind == FIN_OMEGA) {  // <t, s>, ||t||^2
    // t = A s = 0 means s = 0: omega = 0, x += alpha p finishes
    if (n2 != 0.0) S.mvp = mvp;
    S.omega = quot[0];
  } else {  // FIN_RHO: <r_hat, r>, ||r||^2
    const double rnorm = root[0], rel = root[1];
    const double2 beta = cmul(quot[0], quot[1]);
    S.beta = beta;
    S.mbo = cneg(cmul(beta, omega));
    S.rho_old = rho;
    S.rho = d;
    S.rnorm = rnorm;
    S.iters = iters;
    if (hist != nullptr && iters <= hist_len) hist[(long long)r * hist_len + iters - 1] = rel;
    if (rel <= tol)
      status[r] = ST_RECURSIVE;
    else if (iters >= max_iter)
      status[r] = ST_MAXITER;
    else if (vanishes && S.shadows < SHADOWS_MAX) {   // the host loop resets the vectors
      S.shadows += 1;
      reset_recurrence(S, n2);
      status[r] = ST_RESTART;
    } else if (vanishes)
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
