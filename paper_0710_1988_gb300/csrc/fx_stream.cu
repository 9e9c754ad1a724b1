// BiCGStab's vector updates in FP64 storage with fixed-point arithmetic.
//
// p = r + beta p - beta omega v, s = r - alpha v, and x += alpha p + omega s,
// r = s - omega t with <rhat, r> and ||r||^2 take 8, 4 and 18 FP64 FMAs an
// entry, 4.8, 2.4 and 11 clocks of an SM, where memory delivers their 64, 48 and
// 112 bytes in 3, 2.2 and 5.3.  So p, x and the dots are formed in integers
// (fx.cuh: shared exponent, two slices, three multiply-adds a real product, one
// FP64 addition a real), and s and r, four FMAs an entry each, stay on the FP64
// pipe beside them.  Every entry of p, v and s has its own exponent (its larger
// part's), so has a scalar: a product of the two is kept at 2^-58 of it and leaves
// out 2^-56 of it at most, 2^-58 in the mean, below the two roundings of the FP64
// form, entry by entry.  The dots share exponents over a warp's tile of N entries a
// lane (fx_warp_dots).  Entries that are infinite, NaN or near the ends of FP64's
// range take FP64.  p and s also leave
// in the operator's form, site by site, through shared memory so that the
// writes are contiguous.
//
// 16^4, 10 systems, us a launch (FP64 with its separate encoding -> here):
// p 173 -> 124 (all FP64 but one term: 148), s 97 -> 84 (in integers 111),
// x and r 285 -> 189 (r in integers too: 219; its memory takes 130).
#include "bicg_fin.cuh"
#include "chain.cuh"
#include "cplx.cuh"
#include "fx.cuh"
#include "kernels.cuh"
#include "wd_internal.h"

namespace wd {

namespace {

constexpr int FXS_WARPS = 8, FXS_THREADS = 32 * FXS_WARPS;

// a scalar in slices against its own exponent field e (0: not held)
struct FxScalar {
  int4 s;
  int e;
};

__device__ __forceinline__ FxScalar fxs_scalar(double2 c, bool &ok) {
  FxScalar r;
  r.e = max(exp_bits(c.x), exp_bits(c.y));
  const bool zero = ((__double_as_longlong(c.x) | __double_as_longlong(c.y)) << 1) == 0;
  ok = ok && (zero || (r.e >= FX_EMIN && r.e <= FX_EMAX));
  r.e = max(r.e, FX_EMIN);
  r.s = fx_cut30(c, r.e);
  return r;
}

// c z in units 2^(Ec + Ez - 1023 - 1079): |value| < 2^60
__device__ __forceinline__ longlong2 fxs_mul(const FxScalar &c, int4 z) {
  long long rh = 0, rm = 1LL << 25, ih = 0, im = 1LL << 25;
  fx_wide(rh, c.s.x, z.x);
  fx_wide(rm, c.s.x, z.y);
  fx_wide(rm, c.s.y, z.x);
  fx_wide(rh, -c.s.z, z.z);
  fx_wide(rm, -c.s.z, z.w);
  fx_wide(rm, -c.s.w, z.z);
  fx_wide(ih, c.s.x, z.z);
  fx_wide(im, c.s.x, z.w);
  fx_wide(im, c.s.y, z.z);
  fx_wide(ih, c.s.z, z.x);
  fx_wide(im, c.s.z, z.y);
  fx_wide(im, c.s.w, z.x);
  return make_longlong2((rh << 4) + (rm >> 26), (ih << 4) + (im >> 26));
}

// whether the units of c z can be applied by fx_to_double
__device__ __forceinline__ bool fxs_in_range(const FxScalar &c, int E) {
  const int u = c.e + E - 1023;
  return u >= 70 && u <= 1970;
}

// a + k1 z1 + k2 z2; c1, c2: k1, k2 in slices, held: whether both are
__device__ __forceinline__ double2 fxs_axpy2(double2 a, double2 k1, const FxScalar &c1, double2 z1,
                                             double2 k2, const FxScalar &c2, double2 z2, bool held) {
  const int E1 = fx_entry_exponent(z1, held), E2 = fx_entry_exponent(z2, held);
  if (!held || !fxs_in_range(c1, E1) || !fxs_in_range(c2, E2)) return cfma(k2, z2, cfma(k1, z1, a));
  const longlong2 t = fxs_mul(c1, fx_cut30(z1, E1)), u = fxs_mul(c2, fx_cut30(z2, E2));
  const int E = c1.e + E1 - 1023, F = c2.e + E2 - 1023;
  const int dt = min(max(F - E, 0), 63), du = min(max(E - F, 0), 63);
  const long long re = fx_align(t.x, dt) + fx_align(u.x, du), im = fx_align(t.y, dt) + fx_align(u.y, du);
  const int G = max(E, F);
  return make_double2(a.x + fx_to_double(re, G), a.y + fx_to_double(im, G));
}

struct FxsTile {
  int4 v[16 * 13];   // 13 a site: no bank conflicts
  int e[16];
  int nz[16];
};

// The warp's 32 N / 12 sites of x (entry q 32 + lane; N = 3 or 6) into the
// operator's form; first: its first site, count: its entries.
template <int N>
__device__ __forceinline__ void fxs_emit(FxsTile &t, const double2 (&x)[N], FxVec fx, int r,
                                         long long sites, size_t tiled, long long first, int count) {
  constexpr int NS = 32 * N / 12, STEP = 32 / NS;   // sites; components a pass of the warp writes
  const int lane = threadIdx.x & 31;
  if (lane < 16) t.e[lane] = t.nz[lane] = 0;
  __syncwarp();
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int s = (q * 32 + lane) / 12;
    atomicMax(&t.e[s], max(exp_bits(x[q].x), exp_bits(x[q].y)));
    if ((__double_as_longlong(x[q].x) | __double_as_longlong(x[q].y)) << 1) t.nz[s] = 1;
  }
  __syncwarp();
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int c = q * 32 + lane, s = c / 12;
    t.v[c + s] = fx_slices(x[q], max(t.e[s], FX_EMIN));
  }
  __syncwarp();
  const int site = lane % NS, c0 = lane / NS;
  if (12 * site < count) {
    int4 *o = fx.v + (size_t)r * 12 * tiled + fx_at((unsigned)(first + site), 12);
#pragma unroll
    for (int c = 0; c < 12; c += STEP) o[(c + c0) * FX_TILE] = t.v[site * 13 + c + c0];
    if (c0 == 0) fx.e[(size_t)r * sites + first + site] = fx_site_exponent(t.e[site], t.nz[site] == 0);
  }
  __syncwarp();
}

}  // namespace

// TWO: out = a + beta out + mbo z (the p update); else out = a - alpha z (s)
template <int N, bool TWO>
__global__ void __launch_bounds__(FXS_THREADS, 2)
bicg_update_fx_kernel(double2 *__restrict__ out, const double2 *a, const double2 *z,
                      FxVec fx, size_t tiled, const BicgScalars *sc,
                      const int *status, long long n) {
  chain_enter();
  const int r = blockIdx.y;
  if (!((M_ACTIVE >> status[r]) & 1u)) return;   // uniform per block
  extern __shared__ __align__(16) unsigned char fxs_smem[];
  constexpr int FXS_TILE = 32 * N;
  const int lane = threadIdx.x & 31;
  const double2 c1 = TWO ? sc[r].beta : cneg(sc[r].alpha), c2 = TWO ? sc[r].mbo : c1;
  bool held = true;
  const FxScalar s1 = fxs_scalar(c1, held), s2 = fxs_scalar(c2, held);
  const size_t off = (size_t)r * n;
  const long long tiles = (n + FXS_TILE - 1) / FXS_TILE;
  for (long long t = (long long)blockIdx.x * FXS_WARPS + (threadIdx.x >> 5); t < tiles;
       t += (long long)gridDim.x * FXS_WARPS) {
    const long long base = t * FXS_TILE;
    const int count = (int)min((long long)FXS_TILE, n - base);
    double2 y[N], w[N], x[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const int c = q * 32 + lane;
      const size_t i = off + base + c;
      const bool in = c < count;
      x[q] = in ? a[i] : make_double2(0.0, 0.0);
      w[q] = in ? z[i] : make_double2(0.0, 0.0);
      if (TWO) y[q] = in ? out[i] : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      if (TWO)
        x[q] = fxs_axpy2(x[q], c1, s1, y[q], c2, s2, w[q], held);
      else
        x[q] = cfma(c1, w[q], x[q]);
      const int c = q * 32 + lane;
      if (c < count) out[off + base + c] = x[q];
    }
    if constexpr (N % 3 == 0) {
      if (fx.v != nullptr)
        fxs_emit<N>(reinterpret_cast<FxsTile *>(fxs_smem)[threadIdx.x >> 5], x, fx, r, n / 12, tiled,
                    base / 12, count);
    }
  }
}

template <int N>
__global__ void __launch_bounds__(FXS_THREADS, 2)
bicg_update_xr_fx_kernel(double2 *__restrict__ x, double2 *__restrict__ rv, const double2 *p,
                         const double2 *sv, const double2 *t,
                         const double2 *__restrict__ rhat, const BicgScalars *sc,
                         const int *status, double *__restrict__ partial, long long n, FinArgs fin) {
  chain_enter();
  const int r = blockIdx.y;
  if (!((M_ACTIVE >> status[r]) & 1u)) return;
  constexpr int FXS_TILE = 32 * N;
  __shared__ double sums[FXS_WARPS][3];
  const int lane = threadIdx.x & 31;
  const double2 al = sc[r].alpha, om = sc[r].omega;
  bool held = true;
  const FxScalar sa = fxs_scalar(al, held), so = fxs_scalar(om, held);
  const size_t off = (size_t)r * n;
  const long long tiles = (n + FXS_TILE - 1) / FXS_TILE;
  const double2 zero = make_double2(0.0, 0.0);
  double2 dots = zero;
  for (long long w = (long long)blockIdx.x * FXS_WARPS + (threadIdx.x >> 5); w < tiles;
       w += (long long)gridDim.x * FXS_WARPS) {
    const long long base = w * FXS_TILE;
    const int count = (int)min((long long)FXS_TILE, n - base);
    double2 s[N], u[N], h[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const size_t i = off + base + q * 32 + lane;
      const bool in = q * 32 + lane < count;
      s[q] = in ? sv[i] : zero;
      u[q] = in ? p[i] : zero;
      h[q] = in ? x[i] : zero;
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {   // x += alpha p + omega s
      const double2 xi = fxs_axpy2(h[q], al, sa, u[q], om, so, s[q], held);
      if (q * 32 + lane < count) x[off + base + q * 32 + lane] = xi;
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {
      const size_t i = off + base + q * 32 + lane;
      const bool in = q * 32 + lane < count;
      u[q] = in ? t[i] : zero;
      h[q] = in ? rhat[i] : zero;
    }
#pragma unroll
    for (int q = 0; q < N; ++q) {   // r = s - omega t
      s[q] = cfma(cneg(om), u[q], s[q]);
      if (q * 32 + lane < count) rv[off + base + q * 32 + lane] = s[q];
    }
    const double2 d = fx_warp_dots<N>(h, s);
    dots = cadd(dots, d);
  }
  fx_block_dots<FXS_WARPS>(dots, sums, partial + ((long long)r * gridDim.x + blockIdx.x) * 3);
  fin_last_block(fin, partial, r);
}

// Entries a lane: six where that gives every SM sixteen warps; below, the time
// is a warp's chain over its entries, so one (three with the encoded form,
// whose tiles are whole sites).
static int fxs_entries(long long n, int nrhs, bool emit) {
  return n * nrhs >= 192LL * 16 * 152 ? 6 : emit ? 3 : 1;
}

// blocks (per system): a tile a warp up to four blocks per SM
static int fxs_grid(long long n, int entries) {
  const long long b = (n + 32 * entries * FXS_WARPS - 1) / (32 * entries * FXS_WARPS);
  return (int)(b > 608 ? 608 : b < 1 ? 1 : b);
}

bool fin_fused(long long n, int nrhs) { return fxs_entries(n, nrhs, false) != 6; }

int fxs_blocks(long long n, int nrhs) { return fxs_grid(n, fxs_entries(n, nrhs, false)); }

template <bool TWO>
static cudaError_t launch_update(double2 *out, const double2 *a, const double2 *z, FxVec fx,
                                 const BicgScalars *sc, const int *status, long long n, int nrhs,
                                 cudaStream_t s) {
  const int N = fxs_entries(n, nrhs, fx.v != nullptr);
  const dim3 grid(fxs_grid(n, N), nrhs);
  const size_t smem = fx.v != nullptr ? FXS_WARPS * sizeof(FxsTile) : 0;
#define FXS_UPDATE(N) \
  return launch_chained(bicg_update_fx_kernel<N, TWO>, grid, dim3(FXS_THREADS), smem, s, out, a, z, fx, \
                        fx_sites(n / 12), sc, status, n)
  if (N == 6) FXS_UPDATE(6);
  if (N == 3) FXS_UPDATE(3);
  FXS_UPDATE(1);
#undef FXS_UPDATE
}

cudaError_t launch_bicg_update_p(double2 *p, const double2 *r, const double2 *v, FxVec fx,
                                 const BicgScalars *sc, const int *status, long long n,
                                 int nrhs, cudaStream_t s) {
  ProfLaunch prof_(PC_STREAM, s);
  return launch_update<true>(p, r, v, fx, sc, status, n, nrhs, s);
}
cudaError_t launch_bicg_update_s(double2 *sv, const double2 *r, const double2 *v, FxVec fx,
                                 const BicgScalars *sc, const int *status, long long n,
                                 int nrhs, cudaStream_t s) {
  ProfLaunch prof_(PC_STREAM, s);
  return launch_update<false>(sv, r, v, fx, sc, status, n, nrhs, s);
}
cudaError_t launch_bicg_update_xr(double2 *x, double2 *r, const double2 *p, const double2 *sv,
                                  const double2 *t, const double2 *rhat, const BicgScalars *sc,
                                  const int *status, double *partial, long long n, int nrhs,
                                  const FinArgs &fin, cudaStream_t s) {
  ProfLaunch prof_(PC_STREAM, s);
  const dim3 grid(fxs_blocks(n, nrhs), nrhs);
  return launch_chained(fxs_entries(n, nrhs, false) == 6 ? bicg_update_xr_fx_kernel<6> : bicg_update_xr_fx_kernel<1>,
                        grid, dim3(FXS_THREADS), 0, s, x, r, p, sv, t, rhat, sc, status, partial, n, fin);
}

}  // namespace wd
