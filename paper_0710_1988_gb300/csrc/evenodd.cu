// Even-odd preconditioned Wilson operator (Sec. 3 solves "the even-odd
// preconditioned system"; the paper does not write it out):
//
//   A_hat x_e = (1 + i mu gamma5) x_e - kappa^2 D_eo A_oo^{-1} D_oe x_e,
//   A_oo^{-1} = (1 - i mu gamma5) / (1 + mu^2),
//   b_hat = b_e + kappa D_eo A_oo^{-1} b_o,   x_o = A_oo^{-1} (b_o + kappa D_oe x_e).
//
// Half-lattice vectors hold the sites of one parity, compact index s / 2
// (Lx even: the two sites of an x-pair have opposite parities), in the
// boundary spinor layout.  A_hat^dagger = gamma5 A_hat(-mu) gamma5: the hop
// kernels swap projectors and the diagonal terms flip mu, as in dslash.cu.
#include <cmath>

#include "bicg_fin.cuh"
#include "chain.cuh"
#include "cplx.cuh"
#include "fx.cuh"
#include "kernels.cuh"
#include "spin.cuh"
#include "wd_internal.h"

namespace wd {

enum { EO_SCHUR1 = 0, EO_SCHUR2 = 1, EO_AXPY = 2 };

template <bool ADJ>
__device__ __forceinline__ void su3_mul_eo(const double2 *__restrict__ u, const double2 (&h)[6],
                                           double2 (&c)[6]) {
  double2 m[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) m[i] = __ldg(u + i);
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int sp = 0; sp < 2; ++sp) {
      double2 acc = make_double2(0.0, 0.0);
#pragma unroll
      for (int b = 0; b < 3; ++b)
        acc = ADJ ? cfmac(m[3 * b + a], h[3 * sp + b], acc) : cfma(m[3 * a + b], h[3 * sp + b], acc);
      c[3 * sp + a] = acc;
    }
}

template <int MU, int S, bool ADJ>
__device__ __forceinline__ void hop_eo(const double2 *__restrict__ src, const double2 *__restrict__ links,
                                       long long q, long long ql, double2 (&acc)[12]) {
  double2 p[12], h[6], c[6];
  const double2 *ps = src + 12 * (q >> 1);
#pragma unroll
  for (int i = 0; i < 12; ++i) p[i] = __ldg(ps + i);
  project<MU, S>(p, h);
  su3_mul_eo<ADJ>(links + (ql * 4 + MU) * 9, h, c);
  reconstruct<MU, S>(acc, c);
}

// out (parity pout, compact) from h = D_{pout, 1-pout} src:
//  EO_SCHUR1: out = (1 - i mu g5) h / (1 + mu^2)
//  EO_SCHUR2: out = (1 + i mu g5) same - kappa^2 h   (+ reduction epilogue)
//  EO_AXPY:   out = same + kappa h
template <bool DAG, int MODE, int EPI>
__global__ void __launch_bounds__(128)
wilson_eo_kernel(const double2 *__restrict__ links, const double2 *__restrict__ src,
                 const double2 *__restrict__ same, double2 *__restrict__ out, LatticeGeom g,
                 int pout, double kappa, double mu, double inv_1mu2,
                 const double2 *__restrict__ aux,
                 double *__restrict__ partial, const int *__restrict__ status, unsigned mask,
                 unsigned long long *__restrict__ sites) {
  const int r = blockIdx.y;
  if (status != nullptr && !((mask >> status[r]) & 1u)) return;
  if (sites != nullptr && blockIdx.x == 0 && threadIdx.x == 0)
    atomicAdd(sites, (unsigned long long)g.V);  // two half hops = one full MVP of work
  const long long Vh = g.V / 2;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long off = (long long)r * 12 * Vh;
  double red[3] = {0.0, 0.0, 0.0};
  if (i < Vh) {
    // full site of parity pout in the x-pair (2i, 2i+1)
    const long long s0 = 2 * i;
    long long t1 = s0 / g.L[0];
    const int y = (int)(t1 % g.L[1]);
    t1 /= g.L[1];
    const int z = (int)(t1 % g.L[2]);
    const int t = (int)(t1 / g.L[2]);
    const long long s = s0 + (((y + z + t) & 1) != pout ? 1 : 0);
    const Nbrs nb = neighbours(s, g.L);
    constexpr int F = DAG ? +1 : -1;
    constexpr int B = -F;
    const double2 *sr = src + off;
    double2 acc[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) acc[c] = make_double2(0.0, 0.0);
    hop_eo<0, F, false>(sr, links, nb.up[0], s, acc);
    hop_eo<0, B, true>(sr, links, nb.dn[0], nb.dn[0], acc);
    hop_eo<1, F, false>(sr, links, nb.up[1], s, acc);
    hop_eo<1, B, true>(sr, links, nb.dn[1], nb.dn[1], acc);
    hop_eo<2, F, false>(sr, links, nb.up[2], s, acc);
    hop_eo<2, B, true>(sr, links, nb.dn[2], nb.dn[2], acc);
    hop_eo<3, F, false>(sr, links, nb.up[3], s, acc);
    hop_eo<3, B, true>(sr, links, nb.dn[3], nb.dn[3], acc);
    const double tmu = DAG ? -mu : mu;
    double2 *o = out + off + 12 * i;
    double2 sm[12];
    if (MODE != EO_SCHUR1) {
#pragma unroll
      for (int c = 0; c < 12; ++c) sm[c] = __ldg(same + off + 12 * i + c);
    }
    const double inv = inv_1mu2;  // 1 / (1 + mu^2), formed once on the host
    const double k2 = kappa * kappa;
#pragma unroll
    for (int c = 0; c < 12; ++c) {
      const double gm = c < 6 ? tmu : -tmu;  // mu * gamma5 entry
      double2 v;
      if (MODE == EO_SCHUR1) {           // (1 - i mu g5) h / (1 + mu^2)
        v.x = (acc[c].x + gm * acc[c].y) * inv;
        v.y = (acc[c].y - gm * acc[c].x) * inv;
      } else if (MODE == EO_SCHUR2) {    // (1 + i mu g5) same - kappa^2 h
        v.x = fma(-k2, acc[c].x, sm[c].x - gm * sm[c].y);
        v.y = fma(-k2, acc[c].y, sm[c].y + gm * sm[c].x);
      } else {                           // same + kappa h
        v.x = fma(kappa, acc[c].x, sm[c].x);
        v.y = fma(kappa, acc[c].y, sm[c].y);
      }
      o[c] = v;
      if (EPI == EPI_DOT) {
        const double2 a = __ldg(aux + off + 12 * i + c);
        red[0] = fma(a.x, v.x, fma(a.y, v.y, red[0]));
        red[1] = fma(a.x, v.y, fma(-a.y, v.x, red[1]));
        red[2] = fma(v.x, v.x, fma(v.y, v.y, red[2]));
      } else if (EPI == EPI_TSTT) {
        red[0] = fma(v.x, sm[c].x, fma(v.y, sm[c].y, red[0]));
        red[1] = fma(v.x, sm[c].y, fma(-v.y, sm[c].x, red[1]));
        red[2] = fma(v.x, v.x, fma(v.y, v.y, red[2]));
      }
    }
  }
  if (EPI != EPI_NONE) {
    block_sum<3>(red);
    if (threadIdx.x == 0) {
      double *d = partial + ((long long)r * gridDim.x + blockIdx.x) * 3;
      d[0] = red[0];
      d[1] = red[1];
      d[2] = red[2];
    }
  }
}

// ----------------------------------------------------------------- fixed-point form

// fx_exact for D_{pout, 1-pout} src at site s.  whole: src has every site's FP64
// values; else those that fixed point does not hold, and psi, e the others.
template <bool DAG>
__device__ __noinline__ bool hops_mixed(const double2 *src, const int4 *psi, const int *e, bool whole,
                                        const double2 *__restrict__ links, const Nbrs32 nb, unsigned s, int sp,
                                        bool special, int lost, double2 *out) {
  auto ld = [&](unsigned q, int c) {
    const unsigned i = q >> 1;
    if (whole || e[i] == FX_SPECIAL) return src[(size_t)i * 12 + c];
    return fx_decode(psi[fx_at(i, 12) + c * FX_TILE], e[i]);
  };
  return fx_exact<DAG, false>(ld, links, nb.up, nb.dn, s, sp, special, lost, out);
}

constexpr size_t EO_SMEM = 2 * WILSON_SITES / 32 * 2 * sizeof(FxStage);    // two stages a warp

// wilson_eo_kernel's modes with the hops in fixed point (fx.cuh): src is the
// encoded operand, src64 its FP64 values, for EO_SCHUR2 only where it has
// FX_SPECIAL.  EO_SCHUR1 writes the odd vector in fixed point (outfx) for the
// second half hop, and in FP64 (out) the sites that need it: values that fixed
// point does not hold, or components so far below their site's largest that its
// unit would be coarser than FP64's rounding of their terms.
template <bool DAG, int MODE, int EPI>
__global__ void __launch_bounds__(2 * WILSON_SITES, 4)
wilson_eo_fx_kernel(const int4 *__restrict__ L, const double2 *__restrict__ links, FxVec src,
                    const double2 *src64, const double2 *same,
                    double2 *__restrict__ out, FxVec outfx, LatticeGeom g, size_t tiled, int pout,
                    double kappa, double mu, double inv_1mu2, int nrhs,
                    const double2 *__restrict__ aux, double *__restrict__ partial,
                    const int *status, unsigned mask, unsigned long long *__restrict__ sites,
                    FinArgs fin) {
  chain_enter();
  const int r = (int)(blockIdx.x % (unsigned)nrhs);
  const long long sb = blockIdx.x / (unsigned)nrhs;
  if (status != nullptr && !((mask >> status[r]) & 1u)) return;
  if (sites != nullptr && sb == 0 && threadIdx.x == 0)
    atomicAdd(sites, (unsigned long long)g.V);  // two half hops = one full MVP of work
  const unsigned Vh = (unsigned)(g.V / 2);
  const int sp = (threadIdx.x >> 4) & 1;
  const long long at = sb * WILSON_SITES + (threadIdx.x >> 5) * 16 + (threadIdx.x & 15);
  const bool valid = at < Vh;
  const unsigned i = valid ? (unsigned)at : Vh - 1;   // idle lanes repeat the last site
  // the site of parity pout in the x-pair (2i, 2i + 1)
  const unsigned q0 = fast_div(2 * i, g.dm[0], g.dsh[0]);
  const unsigned q1 = fast_div(q0, g.dm[1], g.dsh[1]);
  const unsigned q2 = fast_div(q1, g.dm[2], g.dsh[2]);
  const unsigned yzt = (q0 - q1 * (unsigned)g.L[1]) + (q1 - q2 * (unsigned)g.L[2]) + q2;
  const unsigned s = 2 * i + ((int)(yzt & 1u) != pout ? 1u : 0u);
  const Nbrs32 nb = neighbours32(s, g);
  const int *ev = src.e + (size_t)r * Vh;
  const int4 *psi = src.v + (size_t)r * 12 * tiled;
  int eu[4], ed[4], E = 0;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    eu[m] = ev[nb.up[m] >> 1];
    ed[m] = ev[nb.dn[m] >> 1];
    E = max(E, max(eu[m], ed[m]));
  }
  extern __shared__ __align__(128) unsigned char eo_smem[];
  FxStage *stage = reinterpret_cast<FxStage *>(eo_smem) + 2 * (threadIdx.x >> 5);
  longlong2 up[3], low[3];
  const size_t off = (size_t)r * 12 * Vh;
  const long long first = sb * WILSON_SITES + (threadIdx.x >> 5) * 16;   // the warp's first site
  const size_t base = off + (size_t)first * 12;
  const int count = 12 * (int)max(0LL, min(16LL, (long long)Vh - first));
  const unsigned here = (pout ? Vh : 0u) + i, other = pout ? 0u : Vh;
  const uint2 reach = fx_hops<(DAG ? +1 : -1)>(
      stage, [&](int m, bool fwd) {
        return L + fx_at(fwd ? here : other + (nb.dn[m] >> 1), 36) + m * 9 * FX_TILE;
      },
      [&](int m, bool fwd) { return psi + fx_at((fwd ? nb.up[m] : nb.dn[m]) >> 1, 12); },
      [&](double2 *own) { fx_fetch_own(own, same + base, MODE == EO_SCHUR1 ? 0 : count); }, sp, E, eu,
      ed, up, low);
  const double tmu = DAG ? -mu : mu;
  int bits = 0, least = FX_REACH;
  if (MODE == EO_SCHUR1) {   // a stored site's unit is 2^(bits - 56): terms of 2^-7 of the largest sum
    bits = fx_sum_bits(up, low);
    bits = max(bits, __shfl_xor_sync(0xffffffffu, bits, 16));
    least = max(least, bits - 38);
  }
  const int lost = E != 0 ? fx_lost(reach, least) : 0;   // E = 0: all neighbours are zero
  const bool exact = __any_sync(0xffffffffu, E == FX_SPECIAL || lost != 0);
  if (MODE == EO_SCHUR1 && tmu == 0.0 && !exact) {
    // h itself: the sums' slices, without a way through FP64
    if (valid) {
      int4 *o = outfx.v + (size_t)r * 12 * tiled + fx_at(i, 12);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int2 ux = fx_reslice(up[a].x, bits), uy = fx_reslice(up[a].y, bits);
        const int2 lx = fx_reslice(low[a].x, bits), ly = fx_reslice(low[a].y, bits);
        o[(3 * sp + a) * FX_TILE] = make_int4(ux.x, ux.y, uy.x, uy.y);
        o[(6 + 3 * sp + a) * FX_TILE] = make_int4(lx.x, lx.y, ly.x, ly.y);
      }
      if (sp == 0) outfx.e[(size_t)r * Vh + i] = bits ? E + bits - 57 : 0;
    }
    return;
  }
  // the warp's 16 sites of hop sums through shared memory
  double2 *hop = reinterpret_cast<double2 *>(stage + 1);   // 13 a site: no bank conflicts
  double2 *mine = hop + (threadIdx.x & 15) * 13;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    mine[3 * sp + a] = make_double2(fx_to_double(up[a].x, E), fx_to_double(up[a].y, E));
    mine[6 + 3 * sp + a] = make_double2(fx_to_double(low[a].x, E), fx_to_double(low[a].y, E));
  }
  __syncwarp();
  bool in64 = false;   // the site's sums are FP64's
  if (exact)
    in64 = hops_mixed<DAG>(src64 + off, psi, ev, MODE != EO_SCHUR2, links, nb, s, sp, E == FX_SPECIAL, lost, mine);
  __syncwarp();
  if (MODE == EO_SCHUR1) {   // (1 - i mu g5) h / (1 + mu^2)
    double2 v[6];
    int e = 0;
    unsigned long long any = 0;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const double2 h = mine[(c < 3 ? 0 : 3) + 3 * sp + c];
      const double gm = c < 3 ? tmu : -tmu;
      v[c].x = (h.x + gm * h.y) * inv_1mu2;
      v[c].y = (h.y - gm * h.x) * inv_1mu2;
      e = max(e, max(exp_bits(v[c].x), exp_bits(v[c].y)));
      any |= (unsigned long long)(__double_as_longlong(v[c].x) | __double_as_longlong(v[c].y)) << 1;
    }
    e = max(e, __shfl_xor_sync(0xffffffffu, e, 16));
    any |= __shfl_xor_sync(0xffffffffu, any, 16);
    const int Eo = in64 ? FX_SPECIAL : fx_site_exponent(e, any == 0);
    if (valid) {
      int4 *o = outfx.v + (size_t)r * 12 * tiled + fx_at(i, 12);
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const int comp = (c < 3 ? 0 : 3) + 3 * sp + c;
        o[comp * FX_TILE] = fx_slices(v[c], max(e, FX_EMIN));
        if (Eo == FX_SPECIAL) out[off + (size_t)i * 12 + comp] = v[c];
      }
      if (sp == 0) outfx.e[(size_t)r * Vh + i] = Eo;
    }
    return;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  const double2 *own = reinterpret_cast<const double2 *>(stage);
  double2 dv[6], da[6];   // the epilogue's operands
  const double k2 = kappa * kappa;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const int c = q * 32 + (threadIdx.x & 31);
    if (c < count) {
      const double2 sm = own[c], h = hop[c + c / 12];
      double2 v;
      if (MODE == EO_SCHUR2) {    // (1 + i mu g5) same - kappa^2 h
        double2 d = sm;
        if (tmu != 0.0 || exp_bits(sm.x) == 0x7ff || exp_bits(sm.y) == 0x7ff) {
          const double gm = c % 12 < 6 ? tmu : -tmu;
          d.x = sm.x - gm * sm.y;
          d.y = sm.y + gm * sm.x;
        }
        v.x = fma(-k2, h.x, d.x);
        v.y = fma(-k2, h.y, d.y);
      } else {                    // same + kappa h
        v.x = fma(kappa, h.x, sm.x);
        v.y = fma(kappa, h.y, sm.y);
      }
      out[base + c] = v;
      if (EPI != EPI_NONE) {
        dv[q] = v;
        da[q] = EPI == EPI_DOT ? __ldg(aux + base + c) : sm;
      }
    } else if (EPI != EPI_NONE) {
      dv[q] = da[q] = make_double2(0.0, 0.0);
    }
  }
  if (EPI != EPI_NONE) {  // <aux, out> or <out, same>, and <out, out>
    __shared__ double sums[2 * WILSON_SITES / 32][3];
    double2 d = fx_warp_dots<6>(da, dv);
    if (EPI == EPI_TSTT && (threadIdx.x & 31) == 16) d.x = -d.x;   // <out, same>: the conjugate
    const long long nsb = gridDim.x / (unsigned)nrhs;
    fx_block_dots<2 * WILSON_SITES / 32>(d, sums, partial + ((long long)r * nsb + sb) * 3);
    fin_last_block(fin, partial, r);
  }
}

template <bool DAG, int MODE, int EPI>
static cudaError_t launch_eo_fx1(const wd_context *h, FxVec src, const double2 *src64,
                                 const double2 *same, double2 *out, FxVec outfx, int pout, int nrhs,
                                 const double2 *aux, double *partial, const int *status,
                                 unsigned mask, unsigned long long *cnt, const FinArgs &fin, cudaStream_t s) {
  const unsigned grid = (unsigned)((h->V / 2 + WILSON_SITES - 1) / WILSON_SITES) * (unsigned)nrhs;
  const double inv = 1.0 / std::fma(h->mu, h->mu, 1.0);
  return launch_chained(wilson_eo_fx_kernel<DAG, MODE, EPI>, dim3(grid), dim3(2 * WILSON_SITES), EO_SMEM, s,
                        h->links_fx, h->links, src, src64, same, out, outfx, geom_of(h), fx_sites(h->V / 2),
                        pout, h->kappa, h->mu, inv, nrhs, aux, partial, status, mask, cnt, fin);
}

// Stream-ordered scratch for `count` encoded batches of half vectors; v is
// nullptr when the memory is not there.
struct FxScratch {
  FxVec f[2];
  int4 *buf = nullptr;
  cudaStream_t s;
  FxScratch(const wd_context *h, int nrhs, int count, cudaStream_t stream) : s(stream) {
    if (h->links_fx == nullptr || being_captured(s) || (h->V / 2 + WILSON_SITES - 1) / WILSON_SITES * nrhs > 0x7fffffffLL) return;
    const size_t nv = (size_t)nrhs * fx_sites(h->V / 2), one = nv * 12 * sizeof(int4) + nv * sizeof(int);
    if (cudaMallocFromPoolAsync((void **)&buf, count * one, h->pool, s) != cudaSuccess) {
      cudaGetLastError();
      buf = nullptr;
      return;
    }
    for (int i = 0; i < count; ++i)
      f[i] = FxVec{buf + i * 12 * nv, reinterpret_cast<int *>(buf + count * 12 * nv) + i * nv};
  }
  ~FxScratch() {
    if (buf) cudaFreeAsync(buf, s);
  }
};

int eo_blocks(const wd_context *h) { return (int)((h->V / 2 + WILSON_SITES - 1) / WILSON_SITES); }

template <bool DAG>
static void launch_eo(int mode, int epi, dim3 grid, cudaStream_t s, const wd_context *h,
                      const double2 *src, const double2 *same, double2 *out, int pout,
                      const double2 *aux, double *partial, const int *status, unsigned mask,
                      unsigned long long *cnt) {
  const LatticeGeom g = geom_of(h);
  const double inv = 1.0 / std::fma(h->mu, h->mu, 1.0);  // as the device contracts it
#define EO_LAUNCH(M, E)                                                                   \
  wilson_eo_kernel<DAG, M, E><<<grid, WILSON_SITES, 0, s>>>(h->links, src, same, out, g, pout, h->kappa, \
                                                   h->mu, inv, aux, partial, status, mask, cnt)
  if (mode == EO_SCHUR1) EO_LAUNCH(EO_SCHUR1, EPI_NONE);
  else if (mode == EO_AXPY) EO_LAUNCH(EO_AXPY, EPI_NONE);
  else if (epi == EPI_DOT) EO_LAUNCH(EO_SCHUR2, DAG ? EPI_NONE : EPI_DOT);   // never with DAG
  else if (epi == EPI_TSTT) EO_LAUNCH(EO_SCHUR2, DAG ? EPI_NONE : EPI_TSTT);
  else EO_LAUNCH(EO_SCHUR2, EPI_NONE);
#undef EO_LAUNCH
}

static int ensure_eo_tmp(wd_context *h, int nrhs) {
  const size_t need = (size_t)nrhs * 12 * (h->V / 2);
  if (h->eo_tmp_cap >= need) return 0;
  if (h->eo_tmp) cudaFree(h->eo_tmp);
  h->eo_tmp = nullptr;
  h->eo_tmp_cap = 0;
  if (cudaMalloc(&h->eo_tmp, need * sizeof(double2)) != cudaSuccess) return 1;
  h->eo_tmp_cap = need;
  return 0;
}

// out = A_hat in (or A_hat^dagger in), both even half vectors, with the
// reduction epilogues of the full operator on the second half hop.
cudaError_t launch_schur_f64_epi(const wd_context *hc, const double2 *in, double2 *out, int nrhs,
                                 int dagger, int epi, const double2 *aux, double *partial,
                                 const int *status, cudaStream_t s, unsigned mask,
                                 const FxVec *pre, const FinArgs *fin) {
  const FinArgs none{};
  wd_context *h = const_cast<wd_context *>(hc);
  if (ensure_eo_tmp(h, nrhs)) return cudaErrorMemoryAllocation;
  ProfLaunch prof(PC_DSLASH, s);
  unsigned long long *cnt = prof_site_counter();
  FxScratch fx(h, nrhs, pre ? 1 : 2, s);
  if (fx.buf) {
    const FxVec tmp = fx.f[0], src = pre ? *pre : fx.f[1];
    cudaError_t e = cudaSuccess;
    if (!pre) e = launch_fx_encode(in, src, h->V / 2, nrhs, status, mask, s);
    if (e != cudaSuccess) return e;
#define EO_FX(D, M, E, SRC, SRC64, SAME, OUT, OUTFX, POUT, CNT, FIN)                                \
  launch_eo_fx1<D, M, E>(h, SRC, SRC64, SAME, OUT, OUTFX, POUT, nrhs, aux, partial, status, mask, CNT, \
                         FIN, s)
#define EO_FX_PAIR(D, E)                                                                            \
  {                                                                                                 \
    e = EO_FX(D, EO_SCHUR1, EPI_NONE, src, in, nullptr, h->eo_tmp, tmp, 1, nullptr, none);          \
    return e != cudaSuccess ? e : EO_FX(D, EO_SCHUR2, E, tmp, h->eo_tmp, in, out, tmp, 0, cnt,        \
                                              fin ? *fin : none);                                  \
  }
    if (dagger) EO_FX_PAIR(true, EPI_NONE)
    if (epi == EPI_DOT) EO_FX_PAIR(false, EPI_DOT)
    if (epi == EPI_TSTT) EO_FX_PAIR(false, EPI_TSTT)
    EO_FX_PAIR(false, EPI_NONE)
#undef EO_FX_PAIR
  }
  dim3 grid(eo_blocks(h), nrhs);
  if (dagger) {
    launch_eo<true>(EO_SCHUR1, EPI_NONE, grid, s, h, in, nullptr, h->eo_tmp, 1, nullptr, nullptr, status, mask, nullptr);
    launch_eo<true>(EO_SCHUR2, epi, grid, s, h, h->eo_tmp, in, out, 0, aux, partial, status, mask, cnt);
  } else {
    launch_eo<false>(EO_SCHUR1, EPI_NONE, grid, s, h, in, nullptr, h->eo_tmp, 1, nullptr, nullptr, status, mask, nullptr);
    launch_eo<false>(EO_SCHUR2, epi, grid, s, h, h->eo_tmp, in, out, 0, aux, partial, status, mask, cnt);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || fin == nullptr) return e;
  return launch_bicg_finalize(fin->kind, partial, fin->nb, fin->sc, fin->status, fin->hist, fin->hist_len, nrhs, s);
}

// ----------------------------------------------------------------- split / merge / diagonal

// full [rhs][V][12] <-> halves [rhs][V/2][12] of parity 0 (e) and 1 (o)
__global__ void eo_split_kernel(const double2 *__restrict__ full, double2 *__restrict__ e,
                                double2 *__restrict__ o, LatticeGeom g, int merge) {
  const int r = blockIdx.y;
  const long long Vh = g.V / 2;
  for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < g.V;
       s += (long long)gridDim.x * blockDim.x) {
    long long t1 = s / g.L[0];
    const int x = (int)(s % g.L[0]);
    const int y = (int)(t1 % g.L[1]);
    t1 /= g.L[1];
    const int z = (int)(t1 % g.L[2]);
    const int t = (int)(t1 / g.L[2]);
    double2 *half = ((x + y + z + t) & 1) ? o : e;
    double2 *hp = half + ((long long)r * Vh + (s >> 1)) * 12;
    const long long fo = ((long long)r * g.V + s) * 12;
    if (merge) {
      double2 *f = const_cast<double2 *>(full);
#pragma unroll
      for (int c = 0; c < 12; ++c) f[fo + c] = hp[c];
    } else {
#pragma unroll
      for (int c = 0; c < 12; ++c) hp[c] = full[fo + c];
    }
  }
}

// out = (1 - i mu gamma5) in / (1 + mu^2), half vectors
__global__ void aoo_inv_kernel(const double2 *__restrict__ in, double2 *__restrict__ out,
                               double mu, long long n) {
  const double inv = 1.0 / (1.0 + mu * mu);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const double gm = (i % 12) < 6 ? mu : -mu;
    const double2 v = in[i];
    out[i] = make_double2((v.x + gm * v.y) * inv, (v.y - gm * v.x) * inv);
  }
}

static unsigned grid_for(long long n) {
  long long b = (n + 255) / 256;
  return (unsigned)(b > 1216 ? 1216 : (b < 1 ? 1 : b));
}

// out (parity pout) = same + kappa D src
static cudaError_t launch_eo_axpy(const wd_context *h, const double2 *src, const double2 *same,
                                  double2 *out, int pout, int nrhs, cudaStream_t s) {
  FxScratch fx(h, nrhs, 1, s);
  if (fx.buf) {
    const cudaError_t e = launch_fx_encode(src, fx.f[0], h->V / 2, nrhs, nullptr, M_ALL, s);
    return e != cudaSuccess ? e
                            : launch_eo_fx1<false, EO_AXPY, EPI_NONE>(h, fx.f[0], src, same, out, FxVec{nullptr, nullptr}, pout, nrhs,
                                                                      nullptr, nullptr, nullptr, M_ALL, nullptr, FinArgs{}, s);
  }
  launch_eo<false>(EO_AXPY, EPI_NONE, dim3(eo_blocks(h), nrhs), s, h, src, same, out, pout, nullptr,
                   nullptr, nullptr, M_ALL, nullptr);
  return cudaGetLastError();
}

// b_hat = b_e + kappa D_eo A_oo^{-1} b_o  for nrhs full vectors B
cudaError_t launch_eo_prepare(wd_context *h, const double2 *B, double2 *Bhat, double2 *be,
                              double2 *bo, int nrhs, cudaStream_t s) {
  ProfLaunch prof(PC_STREAM, s);
  const LatticeGeom g = geom_of(h);
  const long long nh = (long long)nrhs * 12 * (h->V / 2);
  eo_split_kernel<<<dim3(grid_for(h->V), nrhs), 256, 0, s>>>(B, be, bo, g, 0);
  aoo_inv_kernel<<<grid_for(nh), 256, 0, s>>>(bo, bo, h->mu, nh);
  return launch_eo_axpy(h, bo, be, Bhat, 0, nrhs, s);
}

// X (full) from x_e: x_o = A_oo^{-1} (b_o + kappa D_oe x_e)
cudaError_t launch_eo_reconstruct(wd_context *h, const double2 *B, const double2 *Xe, double2 *X,
                                  double2 *be, double2 *bo, int nrhs, cudaStream_t s) {
  ProfLaunch prof(PC_STREAM, s);
  const LatticeGeom g = geom_of(h);
  const long long nh = (long long)nrhs * 12 * (h->V / 2);
  eo_split_kernel<<<dim3(grid_for(h->V), nrhs), 256, 0, s>>>(B, be, bo, g, 0);
  const cudaError_t e = launch_eo_axpy(h, Xe, bo, be, 1, nrhs, s);  // be <- b_o + kappa D_oe x_e (odd)
  if (e != cudaSuccess) return e;
  aoo_inv_kernel<<<grid_for(nh), 256, 0, s>>>(be, bo, h->mu, nh);
  eo_split_kernel<<<dim3(grid_for(h->V), nrhs), 256, 0, s>>>(X, const_cast<double2 *>(Xe), bo, g, 1);
  return cudaGetLastError();
}

}  // namespace wd
