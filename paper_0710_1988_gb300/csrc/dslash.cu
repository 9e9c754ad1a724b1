// Wilson-Dirac operator A = 1 - kappa*D + i*mu*gamma5 in FP64 (Sec. 1, Sec. 4).
//
// One thread per (site, right-hand side).  Each of the 8 hops projects the
// neighbour spinor onto the 2-spin subspace of (1 -/+ gamma_mu), multiplies
// the two colour vectors by the link (or its adjoint) and rebuilds the
// lower spin pair from the upper one, so a hop costs 2 SU(3) mat-vecs
// instead of 4.  In the chiral basis gamma_mu = [[0, B], [B^dagger, 0]]
// with B = -i sigma_k (k = x, y, z) and B = 1 (t):
//   (1 - gamma_mu) psi = [h ; -B^dagger h],  h = psi_up - B psi_dn
//   (1 + gamma_mu) psi = [h ; +B^dagger h],  h = psi_up + B psi_dn
// A^dagger = gamma5 A(-mu) gamma5 (gamma5-hermiticity, Sec. 1) swaps the
// two projectors and flips the sign of mu.
//
// Optional fused epilogues write one block-partial (3 doubles) per block for
// the BiCGStab scalars: EPI_DOT   <aux, out>, <out, out>   (aux = r_hat)
//                       EPI_TSTT  <out, in>,  <out, out>
#include "bicg_fin.cuh"
#include "chain.cuh"
#include "cplx.cuh"
#include "wd_internal.h"
#include "kernels.cuh"
#include "fx.cuh"
#include "spin.cuh"

namespace wd {

// chi = U h (ADJ = false) or U^dagger h (ADJ = true), two colour vectors
template <bool ADJ>
__device__ __forceinline__ void su3_mul(const double2 *__restrict__ u, const double2 (&h)[6],
                                        double2 (&c)[6]) {
  double2 m[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) m[i] = __ldg(u + i);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
#pragma unroll
    for (int sp = 0; sp < 2; ++sp) {
      double2 acc = make_double2(0.0, 0.0);
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (ADJ)
          acc = cfmac(m[3 * b + a], h[3 * sp + b], acc);
        else
          acc = cfma(m[3 * a + b], h[3 * sp + b], acc);
      }
      c[3 * sp + a] = acc;
    }
  }
}

__device__ __forceinline__ void load_spinor(const double2 *__restrict__ p, double2 (&v)[12]) {
#pragma unroll
  for (int i = 0; i < 12; ++i) v[i] = __ldg(p + i);
}

// out = init + U^dagger h: the product accumulates onto init in its FMA chain.
__device__ __forceinline__ void su3_adj_mul_acc(const double2 *__restrict__ u,
                                                const double2 (&h)[6], const double2 (&init)[6],
                                                double2 (&out)[6]) {
  double2 m[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) m[i] = __ldg(u + i);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int sp = 0; sp < 2; ++sp) {
      double2 acc = init[3 * sp + a];
#pragma unroll
      for (int b = 0; b < 3; ++b) acc = cfmac(m[3 * b + a], h[3 * sp + b], acc);
      out[3 * sp + a] = acc;
    }
}

// Both hops of direction MU.  With chi_f = U_MU(x) h_f (forward, projector
// sign S) and chi_b = U_MU(x - MU)^dagger h_b (backward, sign -S), the pair
// contributes [chi_f + chi_b ; S B^dagger (chi_f - chi_b)] (the lower spin
// pair of each hop is S or -S times B^dagger of its upper pair).  The sum is
// formed by starting chi_b's FMA chain at chi_f and the difference as
// 2 chi_f - sum, which saves the separate additions of the two hops; FIRST
// assigns instead of accumulating.
template <int MU, int S, bool FIRST>
__device__ __forceinline__ void hop_pair(const double2 *__restrict__ psi,
                                         const double2 *__restrict__ links, long long qf,
                                         long long s, long long qb, double2 (&acc)[12]) {
  double2 sum[6], dif[6];
  {
    double2 p[12], h[6], cf[6];
    load_spinor(psi + 12 * qf, p);
    project<MU, S>(p, h);
    su3_mul<false>(links + (s * 4 + MU) * 9, h, cf);
    load_spinor(psi + 12 * qb, p);
    project<MU, -S>(p, h);
    su3_adj_mul_acc(links + (qb * 4 + MU) * 9, h, cf, sum);
#pragma unroll
    for (int i = 0; i < 6; ++i)
      dif[i] = make_double2(fma(2.0, cf[i].x, -sum[i].x), fma(2.0, cf[i].y, -sum[i].y));
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double2 c0 = dif[a], c1 = dif[3 + a];
    // B^dagger applied to (c0, c1): rows 6+a and 9+a of the lower spin pair
    double2 l6, l9;
    if (MU == 0) {        // B^dagger = (i c1, i c0)
      l6 = cmuli(c1);
      l9 = cmuli(c0);
    } else if (MU == 1) { // (c1, -c0)
      l6 = c1;
      l9 = cneg(c0);
    } else if (MU == 2) { // (i c0, -i c1)
      l6 = cmuli(c0);
      l9 = cmulmi(c1);
    } else {              // (c0, c1)
      l6 = c0;
      l9 = c1;
    }
    if (S < 0) {
      l6 = cneg(l6);
      l9 = cneg(l9);
    }
    if (FIRST) {
      acc[a] = sum[a];
      acc[3 + a] = sum[3 + a];
      acc[6 + a] = l6;
      acc[9 + a] = l9;
    } else {
      acc[a] = cadd(acc[a], sum[a]);
      acc[3 + a] = cadd(acc[3 + a], sum[3 + a]);
      acc[6 + a] = cadd(acc[6 + a], l6);
      acc[9 + a] = cadd(acc[9 + a], l9);
    }
  }
}

template <bool DAG, int EPI>
__global__ void __launch_bounds__(128)
wilson_f64_kernel(const double2 *__restrict__ links, const double2 *__restrict__ in,
                  double2 *__restrict__ out, LatticeGeom g, double kappa, double mu,
                  const double2 *__restrict__ aux, double *__restrict__ partial,
                  const int *__restrict__ status, unsigned mask,
                  unsigned long long *__restrict__ sites) {
  const int r = blockIdx.y;
  if (status != nullptr && !((mask >> status[r]) & 1u)) return;  // uniform per block
  if (sites != nullptr && blockIdx.x == 0 && threadIdx.x == 0)
    atomicAdd(sites, (unsigned long long)g.V);  // work accounting for the profiler
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const double2 *psi = in + (long long)r * 12 * g.V;
  double red[3] = {0.0, 0.0, 0.0};
  if (s < g.V) {
    const Nbrs nb = neighbours(s, g.L);
    const long long xp = nb.up[0], xm = nb.dn[0], yp = nb.up[1], ym = nb.dn[1];
    const long long zp = nb.up[2], zm = nb.dn[2], tp = nb.up[3], tm = nb.dn[3];

    constexpr int F = DAG ? +1 : -1;  // projector sign on forward hops (-F on backward)
    double2 acc[12];
    hop_pair<0, F, true>(psi, links, xp, s, xm, acc);
    hop_pair<1, F, false>(psi, links, yp, s, ym, acc);
    hop_pair<2, F, false>(psi, links, zp, s, zm, acc);
    hop_pair<3, F, false>(psi, links, tp, s, tm, acc);

    double2 p[12];
    load_spinor(psi + 12 * s, p);
    const double tmu = DAG ? -mu : mu;
    double2 *o = out + (long long)r * 12 * g.V + 12 * s;
    const double2 *ax = (EPI == EPI_DOT) ? aux + (long long)r * 12 * g.V + 12 * s : nullptr;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
      double2 v;
      v.x = fma(-kappa, acc[c].x, p[c].x);
      v.y = fma(-kappa, acc[c].y, p[c].y);
      if (tmu != 0.0) {  // + i mu gamma5 psi, gamma5 = diag(1, 1, -1, -1)
        const double m = c < 6 ? tmu : -tmu;
        v.x = fma(-m, p[c].y, v.x);
        v.y = fma(m, p[c].x, v.y);
      }
      o[c] = v;
      if (EPI == EPI_DOT) {  // <aux, out> = sum conj(aux) out
        const double2 a = __ldg(ax + c);
        red[0] = fma(a.x, v.x, red[0]);
        red[0] = fma(a.y, v.y, red[0]);
        red[1] = fma(a.x, v.y, red[1]);
        red[1] = fma(-a.y, v.x, red[1]);
        red[2] = fma(v.x, v.x, red[2]);
        red[2] = fma(v.y, v.y, red[2]);
      } else if (EPI == EPI_TSTT) {  // <out, in> and <out, out>
        red[0] = fma(v.x, p[c].x, red[0]);
        red[0] = fma(v.y, p[c].y, red[0]);
        red[1] = fma(v.x, p[c].y, red[1]);
        red[1] = fma(-v.y, p[c].x, red[1]);
        red[2] = fma(v.x, v.x, red[2]);
        red[2] = fma(v.y, v.y, red[2]);
      }
    }
  }
  if (EPI != EPI_NONE) {
    constexpr int NQ = 3;
    block_sum<NQ>(red);
    if (threadIdx.x == 0) {
      double *dst = partial + ((long long)r * gridDim.x + blockIdx.x) * NQ;
#pragma unroll
      for (int q = 0; q < NQ; ++q) dst[q] = red[q];
    }
  }
}

// ----------------------------------------------------------------- fixed-point form

// Links -> fixed-point slices [tile][mu][entry][32], sites parity by parity
// when all extents are even (g.split), and a check that every link may be used
// so: entries within 1 in modulus (to rounding) and every row and column
// summing to between 0.5 and 2.5 in |re| + |im| (a 3x3 unitary matrix:
// between 1 and sqrt(6)), which bounds the sums of fx.cuh and keeps the
// links' own rounding below FP64's.  *bad counts links that fail.
__global__ void __launch_bounds__(128)
fx_links_kernel(const double2 *__restrict__ U, int4 *__restrict__ L, LatticeGeom g,
                int *__restrict__ bad) {
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  const Nbrs32 nb = neighbours32((unsigned)s, g);
  int4 *l = L + fx_at(g.split ? nb.par * (unsigned)(g.V / 2) + ((unsigned)s >> 1) : (unsigned)s, 36);
  bool ok = true;
  for (int mu = 0; mu < 4; ++mu) {
    double row[3] = {0.0, 0.0, 0.0}, col[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const double2 u = U[(s * 4 + mu) * 9 + i];
      const double a = fabs(u.x), b = fabs(u.y);
      ok = ok && a <= 1.0 + 0x1p-20 && b <= 1.0 + 0x1p-20 && a + b <= 1.5;   // false for NaN
      row[i / 3] += a + b;
      col[i % 3] += a + b;
      const double hr = ok ? rint(u.x * 0x1p30) : 0.0, hi = ok ? rint(u.y * 0x1p30) : 0.0;
      const double lr = ok ? rint(fma(u.x, 0x1p30, -hr) * 0x1p29) : 0.0;
      const double li = ok ? rint(fma(u.y, 0x1p30, -hi) * 0x1p29) : 0.0;
      l[(mu * 9 + i) * FX_TILE] = make_int4((int)hr, (int)lr, (int)hi, (int)li);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i)
      ok = ok && row[i] >= 0.5 && row[i] <= 2.5 && col[i] >= 0.5 && col[i] <= 2.5;
  }
  if (!ok) atomicAdd(bad, 1);
}

// Spinors -> fixed point (fx.cuh), one thread per site and system.
__global__ void __launch_bounds__(128)
fx_encode_kernel(const double2 *__restrict__ in, FxVec out, long long sites, size_t tiled,
                 const int *__restrict__ status, unsigned mask) {
  const int r = blockIdx.y;
  if (status != nullptr && !((mask >> status[r]) & 1u)) return;
  const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= sites) return;
  double2 p[12];
  load_spinor(in + ((long long)r * sites + s) * 12, p);
  int e = 0;
  unsigned long long any = 0;
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    e = max(e, max(exp_bits(p[c].x), exp_bits(p[c].y)));
    any |= (unsigned long long)(__double_as_longlong(p[c].x) | __double_as_longlong(p[c].y)) << 1;
  }
  const int E = fx_site_exponent(e, any == 0);
  out.e[(long long)r * sites + s] = E;
  int4 *o = out.v + (size_t)r * 12 * tiled + fx_at((unsigned)s, 12);
#pragma unroll
  for (int c = 0; c < 12; ++c) o[c * FX_TILE] = fx_slices(p[c], max(e, FX_EMIN));
}

// fx_exact on FP64 spinors; a call, so that the kernel's registers are not its own
template <bool DAG>
__device__ __noinline__ void hops_f64(const double2 *psi, const double2 *__restrict__ links,
                                      const LatticeGeom &g, unsigned s, int sp, bool special, int lost, double2 *out) {
  const Nbrs32 nb = neighbours32(s, g);
  fx_exact<DAG, true>([&](unsigned q, int c) { return psi[(size_t)q * 12 + c]; }, links, nb.up, nb.dn, s, sp,
                      special, lost, out);
}

// wilson_f64_kernel's result with the hops in fixed point; `in` is the
// encoded form of in64.  A block covers 64 sites, two lanes (l, l + 16) a
// site; four fit an SM (16 warps, the registers' limit).  With two of 128 sites
// more of the SM waits for a block's last warp (0.274 against 0.267 ms then, 10
// systems at 16^4).  Blocks are numbered system fastest: the nrhs blocks of one range of
// sites share its links through L2.
constexpr size_t FX_SMEM = 2 * WILSON_SITES / 32 * 2 * sizeof(FxStage);   // two stages a warp

template <bool DAG, int EPI>
__global__ void __launch_bounds__(2 * WILSON_SITES, 4)
wilson_fx_kernel(const int4 *__restrict__ L, const double2 *__restrict__ links, FxVec in,
                 const double2 *in64, double2 *__restrict__ out, LatticeGeom g,
                 size_t tiled, double kappa, double mu, int nrhs, const double2 *__restrict__ aux,
                 double *__restrict__ partial, const int *status, unsigned mask,
                 unsigned long long *__restrict__ sites, FinArgs fin) {
  chain_enter();
  const int r = (int)(blockIdx.x % (unsigned)nrhs);
  const long long sb = blockIdx.x / (unsigned)nrhs;
  if (status != nullptr && !((mask >> status[r]) & 1u)) return;  // uniform per block
  if (sites != nullptr && sb == 0 && threadIdx.x == 0)
    atomicAdd(sites, (unsigned long long)g.V);  // work accounting for the profiler
  const int sp = (threadIdx.x >> 4) & 1;
  const long long at = sb * WILSON_SITES + (threadIdx.x >> 5) * 16 + (threadIdx.x & 15);
  const bool valid = at < g.V;
  const unsigned s = valid ? (unsigned)at : (unsigned)g.V - 1;   // idle lanes repeat the last site
  const size_t V = (size_t)g.V;
  const Nbrs32 nb = neighbours32(s, g);
  const int *ev = in.e + (size_t)r * V;
  int eu[4], ed[4], E = 0;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    eu[m] = ev[nb.up[m]];
    ed[m] = ev[nb.dn[m]];
    E = max(E, max(eu[m], ed[m]));
  }
  extern __shared__ __align__(128) unsigned char fx_smem[];
  FxStage *stage = reinterpret_cast<FxStage *>(fx_smem) + 2 * (threadIdx.x >> 5);
  const long long first = sb * WILSON_SITES + (threadIdx.x >> 5) * 16;   // the warp's first site
  const size_t base = ((size_t)r * V + first) * 12;
  const int count = 12 * (int)max(0LL, min(16LL, g.V - first));
  longlong2 up[3], low[3];
  uint2 reach;
  {
    const int4 *psi = in.v + (size_t)r * 12 * tiled;
    const unsigned half = g.split, odd = (unsigned)(g.V / 2);
    const unsigned here = g.split ? (nb.par ? odd : 0u) + (s >> 1) : s;
    const unsigned other = g.split && !nb.par ? odd : 0u;
    reach = fx_hops<(DAG ? +1 : -1)>(
        stage, [&](int m, bool fwd) {
          return L + fx_at(fwd ? here : other + (nb.dn[m] >> half), 36) + m * 9 * FX_TILE;
        },
        [&](int m, bool fwd) { return psi + fx_at(fwd ? nb.up[m] : nb.dn[m], 12); },
        [&](double2 *own) { fx_fetch_own(own, in64 + base, count); }, sp, E, eu, ed,
        up, low);
  }
  // the warp's 16 sites of hop sums through shared memory, so that its reads
  // and writes of the FP64 vectors are contiguous
  double2 *hop = reinterpret_cast<double2 *>(stage + 1);   // 13 a site: no bank conflicts
  double2 *mine = hop + (threadIdx.x & 15) * 13;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    mine[3 * sp + a] = make_double2(fx_to_double(up[a].x, E), fx_to_double(up[a].y, E));
    mine[6 + 3 * sp + a] = make_double2(fx_to_double(low[a].x, E), fx_to_double(low[a].y, E));
  }
  const int lost = E != 0 ? fx_lost(reach, FX_REACH) : 0;   // E = 0: all neighbours are zero
  __syncwarp();
  if (__any_sync(0xffffffffu, E == FX_SPECIAL || lost != 0))
    hops_f64<DAG>(in64 + (size_t)r * 12 * V, links, g, s, sp, E == FX_SPECIAL, lost, mine);
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  const double2 *own = reinterpret_cast<const double2 *>(stage);
  double2 dv[6], da[6];   // the epilogue's operands
  const double tmu = DAG ? -mu : mu;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const int c = q * 32 + (threadIdx.x & 31);
    if (c < count) {
      const double2 p = own[c], d = hop[c + c / 12];
      double2 v;
      v.x = fma(-kappa, d.x, p.x);
      v.y = fma(-kappa, d.y, p.y);
      if (tmu != 0.0) {  // + i mu gamma5 psi, gamma5 = diag(1, 1, -1, -1)
        const double m = c % 12 < 6 ? tmu : -tmu;
        v.x = fma(-m, p.y, v.x);
        v.y = fma(m, p.x, v.y);
      }
      out[base + c] = v;
      if (EPI != EPI_NONE) {
        dv[q] = v;
        da[q] = EPI == EPI_DOT ? __ldg(aux + base + c) : p;
      }
    } else if (EPI != EPI_NONE) {
      dv[q] = da[q] = make_double2(0.0, 0.0);
    }
  }
  if (EPI != EPI_NONE) {  // <aux, out> or <out, in>, and <out, out>
    __shared__ double sums[2 * WILSON_SITES / 32][3];
    double2 d = fx_warp_dots<6>(da, dv);
    if (EPI == EPI_TSTT && (threadIdx.x & 31) == 16) d.x = -d.x;   // <out, in>: the conjugate
    const long long nsb = gridDim.x / (unsigned)nrhs;
    fx_block_dots<2 * WILSON_SITES / 32>(d, sums, partial + ((long long)r * nsb + sb) * 3);
    fin_last_block(fin, partial, r);
  }
}

// ----------------------------------------------------------------- few sites

// b times 1, i, -1, -i (f = 0 .. 3) added to a, slice by slice
__device__ __forceinline__ int4 fx_add_turned(int4 a, int4 b, int f) {
  const int m1 = f == 1 || f == 2 ? -1 : 0, m2 = f >= 2 ? -1 : 0;   // signs of the real and the imaginary part
  const int rh = f & 1 ? b.z : b.x, rl = f & 1 ? b.w : b.y, ih = f & 1 ? b.x : b.z, il = f & 1 ? b.y : b.w;
  return make_int4(a.x + ((rh ^ m1) - m1), a.y + ((rl ^ m1) - m1), a.z + ((ih ^ m2) - m2),
                   a.w + ((il ^ m2) - m2));
}

__device__ __forceinline__ longlong2 shfl_xor(longlong2 v, int lane) {
  return make_longlong2(__shfl_xor_sync(0xffffffffu, v.x, lane), __shfl_xor_sync(0xffffffffu, v.y, lane));
}

// The same product for few sites, where the time is one warp's chain: lane =
// (site of 2) 16 + (upper spin) 8 + (hop of 8), so a lane encodes one
// neighbour's half of the spins, forms one hop's chi and the eight hops of a
// site are summed over lanes; no encoded copy, one launch.  It issues about
// twice the instructions a site of wilson_fx_kernel.
constexpr int FX_FEW_SITES = 8;   // sites a block, two a warp

// fx_exact in the layout of this kernel: the four lanes of a direction form both
// its hops.  q: the lane's neighbour; reached_by: the lanes whose terms reach the
// lane's component, of colour j.  Returns whether the site's sums are in out.
template <bool DAG>
__device__ __noinline__ bool few_f64(const double2 *psi, const double2 *__restrict__ links, unsigned s, int m, bool fwd,
                                     unsigned q, int sp, unsigned reached_by, int j, bool special, bool lost,
                                     double2 *out) {
  const int lane = threadIdx.x & 31;
  auto ld = [&](unsigned at, int c) { return psi[(size_t)at * 12 + c]; };
  bool need = special;
  if (__any_sync(0xffffffffu, lost && !special)) {
    const int t = fx_terms(ld, links + ((size_t)(fwd ? s : q) * 4 + m) * 9, !fwd, q, sp, m < 2 ? 3 - sp : 2 + sp);
    const unsigned t0 = __ballot_sync(0xffffffffu, t & 1), t1 = __ballot_sync(0xffffffffu, t & 2),
                   t2 = __ballot_sync(0xffffffffu, t & 4);
    need = need || (lost && ((j == 0 ? t0 : j == 1 ? t1 : t2) & reached_by) != 0);
  }
  const unsigned any = __ballot_sync(0xffffffffu, need);
  if (any == 0) return false;
  need = ((any >> (lane & 16)) & 0xffffu) != 0;
  const unsigned other = __shfl_xor_sync(0xffffffffu, q, 1);
  double2 acc[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) acc[c] = make_double2(0.0, 0.0);
  fx_pair_f64<true>(ld, links, m, DAG ? +1 : -1, fwd ? q : other, s, fwd ? other : q, acc);
#pragma unroll
  for (int c = 0; c < 12; ++c) {
#pragma unroll
    for (int o = 2; o <= 4; o <<= 1) {
      acc[c].x += __shfl_xor_sync(0xffffffffu, acc[c].x, o);
      acc[c].y += __shfl_xor_sync(0xffffffffu, acc[c].y, o);
    }
    if ((lane & 15) == c) out[c] = acc[c];
  }
  __syncwarp();
  return need;
}

template <bool DAG, int EPI>
__global__ void __launch_bounds__(16 * FX_FEW_SITES)
wilson_fx_few_kernel(const int4 *__restrict__ L, const double2 *__restrict__ links,
                     const double2 *in, double2 *__restrict__ out, LatticeGeom g,
                     double kappa, double mu, int nrhs, const double2 *__restrict__ aux,
                     double *__restrict__ partial, const int *status, unsigned mask,
                     unsigned long long *__restrict__ sites, FinArgs fin) {
  chain_enter();
  const int r = (int)(blockIdx.x % (unsigned)nrhs);
  const long long sb = blockIdx.x / (unsigned)nrhs;
  if (status != nullptr && !((mask >> status[r]) & 1u)) return;  // uniform per block
  if (sites != nullptr && sb == 0 && threadIdx.x == 0)
    atomicAdd(sites, (unsigned long long)g.V);  // work accounting for the profiler
  const int lane = threadIdx.x & 31, sp = (lane >> 3) & 1, m = (lane >> 1) & 3;
  const bool fwd = !(lane & 1);
  const int local = threadIdx.x >> 4;   // site of the block
  const long long at = sb * FX_FEW_SITES + local;
  const bool valid = at < g.V;
  const unsigned s = valid ? (unsigned)at : (unsigned)g.V - 1;   // idle lanes repeat the last site
  const size_t V = (size_t)g.V;
  // this lane's neighbour
  const unsigned q0 = fast_div(s, g.dm[0], g.dsh[0]), q1 = fast_div(q0, g.dm[1], g.dsh[1]);
  const unsigned t = fast_div(q1, g.dm[2], g.dsh[2]);
  const unsigned x = s - q0 * g.L[0], y = q0 - q1 * g.L[1], z = q1 - t * g.L[2];
  const unsigned pos = m == 0 ? x : m == 1 ? y : m == 2 ? z : t;
  const unsigned ext = m == 0 ? g.L[0] : m == 1 ? g.L[1] : m == 2 ? g.L[2] : g.L[3];
  const unsigned step = (m > 0 ? g.L[0] : 1u) * (m > 1 ? g.L[1] : 1u) * (m > 2 ? g.L[2] : 1u);
  const unsigned q = fwd ? (pos + 1 == ext ? s - pos * step : s + step)
                         : (pos == 0 ? s + (ext - 1) * step : s - step);
  const unsigned ls = fwd ? s : q;                            // the link's site
  const unsigned odd = (x + y + z + t + (fwd ? 0 : 1)) & 1u;  // its parity on even extents
  const int4 *l = L + fx_at(g.split ? odd * (unsigned)(V / 2) + (ls >> 1) : ls, 36) + m * 9 * FX_TILE;
  int4 u[9];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      int4 e = __ldg(l + (fwd ? 3 * a + b : 3 * b + a) * FX_TILE);
      if (!fwd) e = make_int4(e.x, e.y, -e.z, -e.w);   // backward: the adjoint
      u[3 * a + b] = e;
    }
  const double2 *psi = in + ((size_t)r * V + q) * 12;
  const int low_spin = m < 2 ? 3 - sp : 2 + sp;   // fx.cuh
  double2 pu[3], pl[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    pu[b] = psi[3 * sp + b];
    pl[b] = psi[3 * low_spin + b];
  }
  int e = 0;
  unsigned long long any = 0;
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    e = max(max(e, max(exp_bits(pu[b].x), exp_bits(pu[b].y))), max(exp_bits(pl[b].x), exp_bits(pl[b].y)));
    any |= (unsigned long long)(__double_as_longlong(pu[b].x) | __double_as_longlong(pu[b].y) |
                                __double_as_longlong(pl[b].x) | __double_as_longlong(pl[b].y)) << 1;
  }
  // the two lanes of a hop hold the neighbour's four spins between them
  e = max(e, __shfl_xor_sync(0xffffffffu, e, 8));
  any |= __shfl_xor_sync(0xffffffffu, any, 8);
  const int Eq = fx_site_exponent(e, any == 0);
  int E = Eq;
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  constexpr int F = DAG ? +1 : -1;
  const bool plus = fwd == (F > 0);   // the hop's projector is 1 + gamma_mu
  const int P0 = m == 0 ? 1 : m == 1 ? 2 * sp : m == 2 ? 1 + 2 * sp : 2;     // projection of 1 - gamma_mu
  const int R0 = m == 0 ? 1 : m == 1 ? 2 - 2 * sp : m == 2 ? 1 + 2 * sp : 0;  // reconstruction of 1 + gamma_mu
  const int P = plus ? (P0 + 2) & 3 : P0, R = plus ? R0 : (R0 + 2) & 3;
  const int raw = max(e, FX_EMIN);
  FxArg h[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) h[b] = FxArg(fx_add_turned(fx_slices(pu[b], raw), fx_slices(pl[b], raw), P));
  longlong2 up[3], low[3];
  const int d = min(E - Eq, 63);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    FxAcc acc = {0, 1LL << 28, 0, 0, 0, 0};
#pragma unroll
    for (int b = 0; b < 3; ++b) fx_cmac<false>(acc, u[3 * a + b], h[b]);
    const longlong2 chi = fx_value<false>(acc);
    up[a] = make_longlong2(fx_align(chi.x, d), fx_align(chi.y, d));
    const long long re = R & 1 ? up[a].y : up[a].x, im = R & 1 ? up[a].x : up[a].y;
    low[a] = make_longlong2(R == 1 || R == 2 ? -re : re, R >= 2 ? -im : im);
    // x and y hops: the lower spin 3 - sp is the other lane's 2 + sp
    const longlong2 other = shfl_xor(low[a], 8);
    if (m < 2) low[a] = other;
  }
  // sum over the hops: z, t lanes keep the lower spin, x, y lanes the upper
  const bool lower = lane & 4;
  longlong2 sum[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const longlong2 got = shfl_xor(lower ? up[a] : low[a], 4), keep = lower ? low[a] : up[a];
    sum[a] = make_longlong2(keep.x + got.x, keep.y + got.y);
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) {
      const longlong2 v = shfl_xor(sum[a], o);
      sum[a] = make_longlong2(sum[a].x + v.x, sum[a].y + v.y);
    }
  }
  // by colour: the lanes whose terms are long enough (fx.cuh); those of this
  // lane's component are the hops of its spin, or for a lower spin the z and t hops
  // of the upper one that it goes with and the x and y hops of the other
  unsigned term[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int hr = (int)(up[a].x >> 32), hi = (int)(up[a].y >> 32);
    term[a] = __ballot_sync(0xffffffffu, ((hr ^ (hr >> 31)) | (hi ^ (hi >> 31))) >= 1 << (FX_REACH - 1));
  }
  const int j = lane & 3;   // colour of this lane's entry (3: none)
  const unsigned reached_by = (lower ? (sp ? 0xf00fu : 0x0ff0u) : (sp ? 0xff00u : 0x00ffu)) << (lane & 16);
  const bool lost = j < 3 && E != 0 && ((j == 0 ? term[0] : j == 1 ? term[1] : term[2]) & reached_by) == 0;
  const longlong2 T = j == 0 ? sum[0] : j == 1 ? sum[1] : sum[2];
  double2 hop = make_double2(fx_to_double(T.x, E), fx_to_double(T.y, E));
  const int c = 3 * ((lower ? 2 : 0) + sp) + j;
  if (__any_sync(0xffffffffu, E == FX_SPECIAL || lost)) {
    __shared__ double2 exact[FX_FEW_SITES][12];
    if (few_f64<DAG>(in + (size_t)r * 12 * V, links, s, m, fwd, q, sp, reached_by, j, E == FX_SPECIAL, lost,
                     exact[local]) && j < 3)
      hop = exact[local][c];
  }
  double2 dv[1] = {make_double2(0.0, 0.0)}, da[1] = {make_double2(0.0, 0.0)};
  if (valid && j < 3) {
    const size_t i = ((size_t)r * V + s) * 12 + c;
    const double2 p = in[i];
    const double tmu = DAG ? -mu : mu;
    double2 v;
    v.x = fma(-kappa, hop.x, p.x);
    v.y = fma(-kappa, hop.y, p.y);
    if (tmu != 0.0) {  // + i mu gamma5 psi, gamma5 = diag(1, 1, -1, -1)
      const double mm = lower ? -tmu : tmu;
      v.x = fma(-mm, p.y, v.x);
      v.y = fma(mm, p.x, v.y);
    }
    out[i] = v;
    if (EPI != EPI_NONE) {
      dv[0] = v;
      da[0] = EPI == EPI_DOT ? __ldg(aux + i) : p;
    }
  }
  if (EPI != EPI_NONE) {  // <aux, out> or <out, in>, and <out, out>
    __shared__ double sums[FX_FEW_SITES / 2][3];
    double2 dd = fx_warp_dots<1>(da, dv);
    if (EPI == EPI_TSTT && lane == 16) dd.x = -dd.x;   // <out, in>: the conjugate
    const long long nsb = gridDim.x / (unsigned)nrhs;
    fx_block_dots<FX_FEW_SITES / 2>(dd, sums, partial + ((long long)r * nsb + sb) * 3);
    fin_last_block(fin, partial, r);
  }
}

// Whether the few-site kernel serves nrhs systems of the full operator: up to
// where the two forms take the same time, in sites x systems.
// us an apply, this kernel / encoding + wilson_fx_kernel: even extents 4096 8.2 /
// 12.4, 12288 13.9 / 16.1, 14336 15.4 / 16.2, 16384 17.4 / 16.4; with an odd extent,
// where the links are not stored by parity, 3969 8.7 / 14.5, 11979 12.5 / 18.5,
// 20449 18.5 / 20.6, 24167 21.1 / 20.0 (one system; seven to 56 alike).
// us a BiCGStab iteration (epi), whose products come with their input encoded:
// even 4096 49.7 / 54.1, 4608 53.6 / 54.4, 5120 57.7 / 56.6, 8192 68.0 / 65.6; odd 8019
// 67.4 / 68.8, 11025 71.9 / 79.4, 11979 83.6 / 83.6, 14641 92.7 / 83.2.
static bool fx_few(const wd_context *h, int nrhs, int epi) {
  const bool even = geom_of(h).split;
  const long long most = epi != EPI_NONE ? (even ? 4608 : 11264) : even ? 14336 : 21504;
  return !h->eo && h->links_fx != nullptr && h->V * nrhs <= most;
}

// The handle's fixed-point links, or none where they do not fit fx.cuh's
// bounds or the memory, of which they may take a quarter of what is free: the
// FP64 kernel then serves.
cudaError_t fx_links_create(wd_context *h) {
  h->links_fx = nullptr;
  if (h->V >= (1LL << 31)) return cudaSuccess;
  int *bad = nullptr, hbad = 1;
  const size_t bytes = sizeof(int4) * 36 * fx_sites(h->V);
  size_t free_bytes = 0, all = 0;
  if (bytes > ((size_t)64 << 20) && cudaMemGetInfo(&free_bytes, &all) == cudaSuccess && bytes > free_bytes / 4)
    return cudaSuccess;
  if (cudaMalloc(&h->links_fx, bytes) != cudaSuccess) {
    cudaGetLastError();
    h->links_fx = nullptr;
    return cudaSuccess;
  }
  cudaError_t e = cudaMalloc(&bad, sizeof(int));
  if (e == cudaSuccess) e = cudaMemset(bad, 0, sizeof(int));
  if (e == cudaSuccess) {
    fx_links_kernel<<<(unsigned)((h->V + 127) / 128), 128>>>(h->links, h->links_fx, geom_of(h), bad);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost);
  if (bad) cudaFree(bad);
  if (hbad != 0) {
    cudaFree(h->links_fx);
    h->links_fx = nullptr;
  }
  return e;
}

void fx_links_release(wd_context *h) {
  if (h->links_fx == nullptr) return;
  cudaDeviceSynchronize();
  cudaFree(h->links_fx);
  h->links_fx = nullptr;
  if (h->pool) cudaMemPoolTrimTo(h->pool, 0);
  cudaGetLastError();   // of the allocation that failed
}

cudaError_t launch_fx_encode(const double2 *in, FxVec f, long long sites, int nrhs,
                                    const int *status, unsigned mask, cudaStream_t s) {
  fx_encode_kernel<<<dim3((unsigned)((sites + 127) / 128), nrhs), 128, 0, s>>>(in, f, sites, fx_sites(sites), status, mask);
  return cudaGetLastError();
}

static cudaError_t launch_wilson_fx(const wd_context *h, FxVec f, const double2 *in, double2 *out,
                                    int nrhs, int dagger, int epi, const double2 *aux,
                                    double *partial, const int *status, cudaStream_t s,
                                    unsigned mask, unsigned long long *cnt, const FinArgs &fin) {
  const unsigned grid = (unsigned)((h->V + WILSON_SITES - 1) / WILSON_SITES) * (unsigned)nrhs;
  const LatticeGeom g = geom_of(h);
#define WFX(D, E)                                                                                \
  return launch_chained(wilson_fx_kernel<D, E>, dim3(grid), dim3(2 * WILSON_SITES), FX_SMEM, s,      \
                        h->links_fx, h->links, f, in, out, g, fx_sites(h->V), h->kappa, h->mu,   \
                        nrhs, aux, partial, status, mask, cnt, fin)
  if (epi == EPI_DOT) WFX(false, EPI_DOT);
  if (epi == EPI_TSTT) WFX(false, EPI_TSTT);
  if (dagger) WFX(true, EPI_NONE);
  WFX(false, EPI_NONE);
#undef WFX
}

static cudaError_t launch_wilson_fx_few(const wd_context *h, const double2 *in, double2 *out, int nrhs,
                                        int dagger, int epi, const double2 *aux, double *partial,
                                        const int *status, cudaStream_t s, unsigned mask,
                                        unsigned long long *cnt, const FinArgs &fin) {
  const unsigned grid = (unsigned)((h->V + FX_FEW_SITES - 1) / FX_FEW_SITES) * (unsigned)nrhs;
  const LatticeGeom g = geom_of(h);
#define WFEW(D, E)                                                                              \
  return launch_chained(wilson_fx_few_kernel<D, E>, dim3(grid), dim3(16 * FX_FEW_SITES), 0, s,  \
                        h->links_fx, h->links, in, out, g, h->kappa, h->mu, nrhs, aux, partial, \
                        status, mask, cnt, fin)
  if (epi == EPI_DOT) WFEW(false, EPI_DOT);
  if (epi == EPI_TSTT) WFEW(false, EPI_TSTT);
  if (dagger) WFEW(true, EPI_NONE);
  WFEW(false, EPI_NONE);
#undef WFEW
}

LatticeGeom geom_of(const wd_context *h) {
  LatticeGeom g;
  for (int i = 0; i < 4; ++i) g.L[i] = h->dims[i];
  g.V = h->V;
  for (int i = 0; i < 3; ++i) {
    const unsigned long long d = (unsigned long long)h->dims[i];
    int l = 0;
    while ((1ULL << l) < d) ++l;
    g.dsh[i] = 31 + l;
    g.dm[i] = (1ULL << g.dsh[i]) / d + 1;
  }
  g.split = 1;
  for (int i = 0; i < 4; ++i) g.split &= h->dims[i] % 2 == 0;
  return g;
}

int eo_blocks(const wd_context *h);
cudaError_t launch_schur_f64_epi(const wd_context *h, const double2 *in, double2 *out, int nrhs,
                                 int dagger, int epi, const double2 *aux, double *partial,
                                 const int *status, cudaStream_t s, unsigned mask,
                                 const FxVec *pre, const FinArgs *fin);

bool being_captured(cudaStream_t s) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &st) != cudaSuccess) cudaGetLastError();   // the legacy stream beside a capture
  return st != cudaStreamCaptureStatusNone;
}

int wilson_blocks(const wd_context *h, int nrhs) {
  if (fx_few(h, nrhs, EPI_DOT)) return (int)((h->V + FX_FEW_SITES - 1) / FX_FEW_SITES);
  return h->eo ? eo_blocks(h) : (int)((h->V + WILSON_SITES - 1) / WILSON_SITES);
}

bool wilson_takes_encoded(const wd_context *h, int nrhs) {
  return h->links_fx != nullptr && !fx_few(h, nrhs, EPI_DOT);
}

cudaError_t launch_wilson_f64_epi(const wd_context *h, const double2 *in, double2 *out,
                                  int nrhs, int dagger, int epi, const double2 *aux,
                                  double *partial, const int *status, cudaStream_t s,
                                  unsigned mask, const FxVec *pre, const FinArgs *fin) {
  const FinArgs f = fin ? *fin : FinArgs{};
  if (dagger && epi != EPI_NONE) return cudaErrorInvalidValue;   // no solver iterates A^dagger
  if (h->eo)  // even-odd Schur operator on even half vectors
    return launch_schur_f64_epi(h, in, out, nrhs, dagger, epi, aux, partial, status, s, mask, pre, fin);
  ProfLaunch prof(PC_DSLASH, s);
  unsigned long long *cnt = prof_site_counter();
  if (fx_few(h, nrhs, epi))
    return launch_wilson_fx_few(h, in, out, nrhs, dagger, epi, aux, partial, status, s, mask, cnt, f);
  if (h->links_fx != nullptr && (long long)wilson_blocks(h, nrhs) * nrhs <= 0x7fffffffLL) {
    if (pre != nullptr)
      return launch_wilson_fx(h, *pre, in, out, nrhs, dagger, epi, aux, partial, status, s, mask, cnt, f);
    // scratch for the encoded input, stream-ordered; without it the FP64 kernel
    const size_t nv = (size_t)nrhs * fx_sites(h->V);
    int4 *buf = nullptr;
    if (!being_captured(s) &&
        cudaMallocFromPoolAsync((void **)&buf, nv * (12 * sizeof(int4) + sizeof(int)), h->pool, s) == cudaSuccess) {
      const FxVec enc{buf, reinterpret_cast<int *>(buf + 12 * nv)};
      cudaError_t e = launch_fx_encode(in, enc, h->V, nrhs, status, mask, s);
      if (e == cudaSuccess)
        e = launch_wilson_fx(h, enc, in, out, nrhs, dagger, epi, aux, partial, status, s, mask, cnt, f);
      cudaError_t e2 = cudaFreeAsync(buf, s);
      return e != cudaSuccess ? e : e2;
    }
    cudaGetLastError();
  }
  dim3 grid(wilson_blocks(h, nrhs), nrhs);
  LatticeGeom g = geom_of(h);
#define W64(D, E)                                                                                        \
  wilson_f64_kernel<D, E><<<grid, WILSON_SITES, 0, s>>>(h->links, in, out, g, h->kappa, h->mu, aux, partial, \
                                                        status, mask, cnt)
  if (epi == EPI_DOT) W64(false, EPI_DOT);
  else if (epi == EPI_TSTT) W64(false, EPI_TSTT);
  else if (dagger) W64(true, EPI_NONE);
  else W64(false, EPI_NONE);
#undef W64
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || fin == nullptr) return e;
  return launch_bicg_finalize(f.kind, partial, f.nb, f.sc, f.status, f.hist, f.hist_len, nrhs, s);
}

cudaError_t launch_wilson_f64(const wd_context *h, const double2 *in, double2 *out, int nrhs,
                              int dagger, cudaStream_t s) {
  return launch_wilson_f64_epi(h, in, out, nrhs, dagger, EPI_NONE, nullptr, nullptr, nullptr, s,
                               M_ALL);
}

}  // namespace wd
