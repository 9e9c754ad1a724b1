// Block fixed point for the FP64 Wilson operator.
//
// This GPU issues 1.7 FP64 FMAs per clock and SM (DFMA probe), so a site
// update's ~930 FP64 instructions take 550 clocks of its SM; integer
// multiply-adds of 32 x 32 + 64 bits go at 60 (27 to 35 reached inside these
// kernels), 32-bit integer adds at 120.  The hops' products are therefore formed in integers.  A spinor site
// (24 reals) shares the largest exponent field E of its entries and holds
// each as X = round(x 2^(1078 - E)), |X| <= 2^56: entries down to 2^-3 of the
// site's largest are held exactly, smaller ones to 2^-57 of it.  X is stored
// as two signed slices, X = hi 2^29 + lo with |lo| <= 2^28, |hi| <= 2^27, so
// that a spin projection and the sums and differences of a complex product
// add slices without carries (|hi| <= 2^29, |lo| <= 2^30).  A link entry is
// u = uh 2^-30 + ul 2^-59, |ul| <= 2^28.
//
//   u x = [uh hi + (uh lo + ul hi) 2^-29] 2^(E - 1079)  (+ ul lo 2^-58, left
//         out: below half a unit of X)
//
// takes three multiply-adds per real product, exact in 64-bit sums: with
// every row and column of a link summing to at most 2.5 in |re| + |im| (3x3
// unitary: sqrt(6)), one hop's component is below 2.5 * 2^58 units, the sum
// over the eight hops below 2^62.4 and the middle sums below 2^63.  A sum
// over hops is aligned to the largest E of the neighbours and rounded once
// to FP64 at the end.  Its error is a few units of 2^-57 of the largest
// neighbour entry; the eight hops' FP64 roundings leave more (2-norm against
// 64-bit torch arithmetic, whose own rounding is in both: 1.0e-16 against
// 1.1e-16).  That holds for a component whose own terms are of the size of the
// largest entry.  A component that only smaller entries reach (colours that a
// diagonal link does not mix, spins that a large neighbour's projector leaves out)
// would keep fewer bits than in FP64: fx_hops tells the terms' size, and
// components whose terms all lie below 2^52 units, where FP64 would leave less
// than a few units, are formed in FP64 (fx_exact).
#pragma once

#include <cuda_runtime.h>

#include "cplx.cuh"
#include "spin.cuh"

namespace wd {

// Layout: tiles of 32 sites, [tile][component][32] (12 components of a
// spinor, 4 x 9 entries of a site's links), so that a warp's loads of one
// component are contiguous and the components lie at fixed offsets.
constexpr int FX_TILE = 32;
__device__ __forceinline__ size_t fx_at(unsigned s, unsigned comps) {
  return (size_t)(s >> 5) * (FX_TILE * comps) + (s & 31);
}
inline size_t fx_sites(long long sites) { return (size_t)((sites + FX_TILE - 1) / FX_TILE * FX_TILE); }

constexpr int FX_SPECIAL = 0x7fffffff;   // a site whose FP64 values must be used
constexpr int FX_EMIN = 200, FX_EMAX = 1900;

__device__ __forceinline__ int exp_bits(double x) {
  return (__double2hiint(x) >> 20) & 0x7ff;
}

// shared exponent of a site from the largest exponent field of its entries:
// E for values in range, 0 for a site of zeros, FX_SPECIAL for infinities,
// NaN and magnitudes near the ends of FP64's range.  allzero: every entry is 0.
__device__ __forceinline__ int fx_site_exponent(int emax, bool allzero) {
  if (emax >= FX_EMIN && emax <= FX_EMAX) return emax;
  return allzero ? 0 : FX_SPECIAL;
}

// Slices of x against a shared exponent E >= FX_EMIN, x's own exponent field
// at most E (zeros and subnormals give 0): hi 2^LO + lo = |x| 2^(1049 + LO - E)
// with the sign on both, |lo| <= 2^(LO - 1).  LO = 29: rounded, the form above;
// LO = 30: cut off at its last bit (2^-57 of the largest), without spin
// projections and complex sums the middle products then still fit.  About 17
// instructions; the shift saturates (PTX), so E needs no clamp.
template <int LO>
__device__ __forceinline__ int2 fx_cut(double x, int E) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const unsigned be = (h >> 20) & 0x7ffu;
  const unsigned long long t = ((unsigned long long)((h & 0xfffffu) | 0x100000u) << 32 | l) << 11;
  unsigned long long Y;
  asm("shr.u64 %0, %1, %2;" : "=l"(Y) : "l"(t), "r"((unsigned)E - be + 7u));
  if (LO == 29) Y = (Y + 1) >> 1;
  const int lo = (int)((unsigned)Y << (32 - LO)) >> (32 - LO);
  const int hi = (int)((Y + (1ULL << (LO - 1))) >> LO);
  const int s = (int)h >> 31;
  return make_int2((hi ^ s) - s, (lo ^ s) - s);
}

__device__ __forceinline__ int2 fx_slices(double x, int E) { return fx_cut<29>(x, E); }

__device__ __forceinline__ int4 fx_slices(double2 x, int E) {
  const int2 a = fx_slices(x.x, E), b = fx_slices(x.y, E);
  return make_int4(a.x, a.y, b.x, b.y);
}

__device__ __forceinline__ int4 fx_cut30(double2 x, int E) {
  const int2 a = fx_cut<30>(x.x, E), b = fx_cut<30>(x.y, E);
  return make_int4(a.x, a.y, b.x, b.y);
}

// T 2^(E - 1079) rounded to FP64 (halves away from zero), |T| < 2^63,
// 70 <= E <= 1970
__device__ __forceinline__ double fx_to_double(long long T, int E) {
  const long long s = T >> 63;
  const unsigned long long a = (unsigned long long)((T ^ s) - s);
  const int lz = __clzll((long long)a);                       // 1 .. 64
  const unsigned long long m = ((a << (lz - 1)) + 0x200) >> 10;   // top bit at 52, or 53 after a carry
  const unsigned hi = (unsigned)(m >> 32) + (((unsigned)E + 6u - (unsigned)lz) << 20);
  return __hiloint2double((int)(a == 0 ? 0u : hi | ((unsigned)s & 0x80000000u)), (int)(unsigned)m);
}

// acc += a b: one 32 x 32 + 64-bit multiply-add.  (Sums of products written in
// C are taken apart into more instructions; only fx_mac below is the faster
// for it.)
__device__ __forceinline__ void fx_wide(long long &acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// T 2^(E - 1079) for any E
__device__ __forceinline__ double fx_scaled(long long T, int E) {
  return E >= 70 && E <= 1970 ? fx_to_double(T, E) : ldexp((double)T, E - 1079);
}

// X 2^(E - 1078) of a stored site's component
__device__ __forceinline__ double2 fx_decode(int4 v, int E) {
  const long long re = ((long long)v.x << 29) + v.y, im = ((long long)v.z << 29) + v.w;
  return make_double2(fx_to_double(re, E + 1), fx_to_double(im, E + 1));
}

// Sums T 2^(E - 1079) of a site, shared by the lanes l and l + 16 (six complex
// components each), as slices of X 2^(E' - 1078): returns E'.  bits: the
// bit length of the largest |T| of the site.
__device__ __forceinline__ int fx_sum_bits(const longlong2 (&a)[3], const longlong2 (&b)[3]) {
  unsigned long long m = 0;
#pragma unroll
  for (int i = 0; i < 3; ++i)
    m |= (unsigned long long)(a[i].x ^ (a[i].x >> 63)) | (unsigned long long)(a[i].y ^ (a[i].y >> 63)) |
         (unsigned long long)(b[i].x ^ (b[i].x >> 63)) | (unsigned long long)(b[i].y ^ (b[i].y >> 63));
  return 64 - __clzll((long long)m);
}

__device__ __forceinline__ int2 fx_reslice(long long T, int bits) {
  const int k = bits - 56;
  const long long X = k > 0 ? (T + (1LL << (k - 1))) >> k : T << -k;
  const int lo = ((int)(unsigned)X << 3) >> 3;
  return make_int2((int)((X - lo) >> 29), lo);
}

// Sums of one complex product chain U h in three real products each (Gauss):
// with U = a + i b, h = c + i d,
//   k1 = (a + b) c, k2 = a (d - c), k3 = b (c + d): U h = (k1 - k3) + i (k1 + k2),
// and with a - b in k1, conj(U) h = (k1 + k3) + i (k1 + k2).  Each real product
// adds its high part and its two middle parts.
struct FxAcc {
  long long h1, m1, h2, m2, h3, m3;
};

// h as (c, d - c, c + d), each (hi, lo)
struct FxArg {
  int2 c, m, p;
  __device__ __forceinline__ FxArg() {}
  __device__ __forceinline__ explicit FxArg(int4 v)
      : c(make_int2(v.x, v.y)), m(make_int2(v.z - v.x, v.w - v.y)), p(make_int2(v.x + v.z, v.y + v.w)) {}
};

__device__ __forceinline__ void fx_mac(long long &h, long long &m, int uh, int ul, int2 x) {
  h += (long long)uh * x.x;
  m += (long long)uh * x.y;
  m += (long long)ul * x.x;
}

template <bool CONJ>
__device__ __forceinline__ void fx_cmac(FxAcc &s, int4 u, const FxArg &x) {
  fx_mac(s.h1, s.m1, CONJ ? u.x - u.z : u.x + u.z, CONJ ? u.y - u.w : u.y + u.w, x.c);
  fx_mac(s.h2, s.m2, u.x, u.y, x.m);
  fx_mac(s.h3, s.m3, u.z, u.w, x.p);
}

template <bool CONJ>
__device__ __forceinline__ longlong2 fx_value(const FxAcc &s) {   // m1 starts at 2^28: rounded
  const long long rm = CONJ ? s.m1 + s.m3 : s.m1 - s.m3, im = s.m1 + s.m2;
  return make_longlong2((CONJ ? s.h1 + s.h3 : s.h1 - s.h3) + (rm >> 29), s.h1 + s.h2 + (im >> 29));
}

// round((x) 2^-d) for 0 <= d <= 63, |x| < 2^62
__device__ __forceinline__ long long fx_align(long long x, int d) {
  return (x + (long long)((1ULL << d) >> 1)) >> d;
}

// a + f b for a factor f = 1, i, -1, -i (F = 0, 1, 2, 3), slice by slice
template <int F>
__device__ __forceinline__ int4 fx_add(int4 a, int4 b) {
  if (F == 0) return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
  if (F == 1) return make_int4(a.x - b.z, a.y - b.w, a.z + b.x, a.w + b.y);
  if (F == 2) return make_int4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
  return make_int4(a.x + b.z, a.y + b.w, a.z - b.x, a.w - b.y);
}

template <int F>
__device__ __forceinline__ longlong2 fx_add(longlong2 a, longlong2 b) {
  if (F == 0) return make_longlong2(a.x + b.x, a.y + b.y);
  if (F == 1) return make_longlong2(a.x - b.y, a.y + b.x);
  if (F == 2) return make_longlong2(a.x - b.x, a.y - b.y);
  return make_longlong2(a.x + b.y, a.y - b.x);
}

// One hop is shared by two lanes of a warp, one per upper spin sp: with h_sp =
// psi_sp + S (B psi)_sp the lane forms chi_sp = U h_sp and adds it to the
// output's spin sp and, times S B^dagger, to one lower spin (spin.cuh): LOW =
// 3 - sp for mu = x, y and 2 + sp for mu = z, t, the one its h_sp came from.
// The factors of sp = 0 and 1 are equal (x, t) or opposite (y, z):
//   projection, S = -1:      x: i   y: sgn   z: i sgn   t: -1    sgn = 1 - 2 sp
//   reconstruction, S = +1:  x: i   y: -sgn  z: i sgn   t:  1
// Splitting a site over two lanes halves its registers (128 at four warps per
// scheduler; one lane a site spills) and its chain, and both read one link.
template <int MU, int S>
struct FxSpin {
  static constexpr bool SGN = MU == 1 || MU == 2;
  static constexpr int P0 = MU == 0 || MU == 2 ? 1 : MU == 1 ? 0 : 2;   // without sgn
  static constexpr int R0 = MU == 0 || MU == 2 ? 1 : MU == 1 ? 2 : 0;
  static constexpr int P = S < 0 ? P0 : (P0 + 2) & 3;
  static constexpr int R = S > 0 ? R0 : (R0 + 2) & 3;
};

// A hop's operands staged in shared memory for the 16 sites of a warp.
struct FxStage {
  int4 u[9][16];      // the link's entries
  int4 psi[12][16];   // the neighbour's components
};

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;"
               ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// Both lanes of a site copy its operands: l, q: the link's and the
// neighbour's first component.
__device__ __forceinline__ void fx_fetch(FxStage &st, const int4 *l, const int4 *q) {
  const int site = threadIdx.x & 15, half = (threadIdx.x >> 4) & 1;
#pragma unroll
  for (int c = 0; c < 12; c += 2) cp_async16(&st.psi[c + half][site], q + (c + half) * FX_TILE);
#pragma unroll
  for (int c = 0; c < 8; c += 2) cp_async16(&st.u[c + half][site], l + (c + half) * FX_TILE);
  if (half == 0) cp_async16(&st.u[8][site], l + 8 * FX_TILE);
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// The warp copies its epilogue's operand, count entries from x.
__device__ __forceinline__ void fx_fetch_own(double2 *own, const double2 *x, int count) {
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const int c = q * 32 + (threadIdx.x & 31);
    if (c < count) cp_async16(own + c, x + c);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// The lane's part of one hop, in units 2^(Eq + d - 1079): up += chi, low +=
// (factor without sgn) chi, low lying in the neighbour's spin cl.  reach: the
// high words of the forward hops' |chi|, or-ed, by colour: four hops tell the terms'
// size, at half the cost of eight (10-system apply at 16^4: 266 us, eight 271, none 257).
template <int MU, int S, bool ADJ>
__device__ __forceinline__ void fx_hop(const FxStage &st, int sp, int cl, int d,
                                       longlong2 (&up)[3], longlong2 (&low)[3], int (&reach)[3]) {
  using W = FxSpin<MU, S>;
  const int site = threadIdx.x & 15, sgn = 1 - 2 * sp;
  const long long half = (long long)((1ULL << d) >> 1);
  FxArg h[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    int4 q = st.psi[3 * cl + b][site];
    if (W::SGN) q = make_int4(sgn * q.x, sgn * q.y, sgn * q.z, sgn * q.w);
    h[b] = FxArg(fx_add<W::P>(st.psi[3 * sp + b][site], q));
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    FxAcc s = {half, 1LL << 28, 0, 0, 0, 0};
#pragma unroll
    for (int b = 0; b < 3; ++b) fx_cmac<ADJ>(s, st.u[ADJ ? 3 * b + a : 3 * a + b][site], h[b]);
    longlong2 chi = fx_value<ADJ>(s);
    chi = make_longlong2(chi.x >> d, chi.y >> d);   // rounded: half is in h1, so in both parts
    const int hr = (int)(chi.x >> 32), hi = (int)(chi.y >> 32);
    if (!ADJ) reach[a] |= (hr ^ (hr >> 31)) | (hi ^ (hi >> 31));
    up[a] = fx_add<0>(up[a], chi);
    low[a] = fx_add<W::R>(low[a], chi);
  }
}

// bit lengths of three words, a byte each
__device__ __forceinline__ unsigned fx_lengths(const int (&m)[3]) {
  return (32u - __clz(m[0])) | (32u - __clz(m[1])) << 8 | (32u - __clz(m[2])) << 16;
}

constexpr int FX_REACH = 21;   // least bit length of a high word: terms of 2^52 units

// The lane's components whose terms are all shorter than `least`, as bits: up's
// colours 0 .. 2, low's 3 .. 5.
__device__ __forceinline__ int fx_lost(uint2 reach, int least) {
  int lost = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lost |= (int)((reach.x >> (8 * a)) & 0xffu) < least ? 1 << a : 0;
    lost |= (int)((reach.y >> (8 * a)) & 0xffu) < least ? 8 << a : 0;
  }
  return lost;
}

// The eight hops of a site for one lane: up is the sum's spin sp, low its
// spin 2 + sp, in units 2^(E - 1079).  The next hop's operands are copied to
// shared memory (st: two stages of this warp) while one hop is computed: the
// copies wait for L2 and hold no registers (through L1, which serves a third
// of them).  A 10-system apply at 16^4 took 0.301 ms with plain loads, 0.332 with
// copies past L1, 0.288 so, of which 0.237 without any copy; with a hop's shift
// rounded in its first sum (no additions, no branch for d = 0) and blocks of
// half the size 0.267, with the epilogue's operand copied during the last hop
// (tail) 0.257, with the terms' lengths (reach) 0.266.  Now the LSU's data pipe (82 %
// of its wavefronts) and the multiply-adds (59 %) bound it, at the 16 warps an SM that
// 128 registers leave.
// The y and z hops come first in their lower sums, whose factor sgn is then
// applied once; between them the lanes exchange the x and y hops' lower sums,
// which belong to the other.  Returned: the bit lengths of the high words of the
// largest forward |chi| in each component's sum, by colour a byte: .x of up, .y of
// low.  On fields whose sites are of one size a component's four stay below 2^52 units
// once in 1e8 sites; where one neighbour exceeds the others by 2^4 or more some per
// cent of the sites go to FP64.
template <int F, class LinkAt, class SiteAt, class Tail>
__device__ __forceinline__ uint2 fx_hops(FxStage *st, LinkAt link, SiteAt site, Tail tail, int sp, int E,
                                         const int (&eu)[4], const int (&ed)[4],
                                         longlong2 (&up)[3], longlong2 (&low)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) up[a] = low[a] = make_longlong2(0, 0);
  int reach[3] = {0, 0, 0};
#define FX_FETCH(B, M, FWD) fx_fetch(st[B], link(M, FWD), site(M, FWD));
#define FX_READY(N)                                            \
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); \
  __syncwarp();
#define FX_SIGN                                                                                    \
  if (sp) {                                                                                        \
    _Pragma("unroll") for (int a = 0; a < 3; ++a) low[a] = make_longlong2(-low[a].x, -low[a].y);   \
  }
#define FX_PAIR(M, CL, NEXT, WAIT)                                      \
  FX_FETCH(1, M, false)                                                 \
  FX_READY(1)                                                           \
  fx_hop<M, F, false>(st[0], sp, CL, min(E - eu[M], 63), up, low, reach); \
  __syncwarp();                                                         \
  NEXT                                                                  \
  FX_READY(WAIT)                                                        \
  fx_hop<M, -F, true>(st[1], sp, CL, min(E - ed[M], 63), up, low, reach); \
  __syncwarp();
  FX_FETCH(0, 1, true)
  FX_PAIR(1, 3 - sp, FX_FETCH(0, 0, true), 1)
  FX_SIGN
  FX_PAIR(0, 3 - sp, FX_FETCH(0, 2, true), 1)
#pragma unroll
  for (int a = 0; a < 3; ++a)
    low[a] = make_longlong2(__shfl_xor_sync(0xffffffffu, low[a].x, 16),
                            __shfl_xor_sync(0xffffffffu, low[a].y, 16));
  const unsigned xy = fx_lengths(reach);
  reach[0] = reach[1] = reach[2] = 0;
  FX_SIGN
  FX_PAIR(2, 2 + sp, FX_FETCH(0, 3, true), 1)
  FX_SIGN
  FX_PAIR(3, 2 + sp, tail(reinterpret_cast<double2 *>(&st[0]));, 1)
  const unsigned zt = fx_lengths(reach);
  return make_uint2(__vmaxu4(xy, zt), __vmaxu4(zt, __shfl_xor_sync(0xffffffffu, xy, 16)));
#undef FX_PAIR
#undef FX_SIGN
#undef FX_READY
#undef FX_FETCH
}

// ----------------------------------------------------------------- in FP64

__device__ __forceinline__ double2 fx_turned(double2 b, int f) {   // i^f b
  const double x = f & 1 ? b.y : b.x, y = f & 1 ? b.x : b.y;
  return make_double2(f == 1 || f == 2 ? -x : x, f >= 2 ? -y : y);
}

// Which colours of the half spinor U h_sp have a nonzero term, h_sp from the
// spins sp and cl of site q: bits 0 .. 2.  ld(q, c): component c of site q.
template <class Load>
__device__ __forceinline__ int fx_terms(Load ld, const double2 *u, bool adj, unsigned q, int sp, int cl) {
  auto nonzero = [](double2 z) {
    return ((__double_as_longlong(z.x) | __double_as_longlong(z.y)) << 1) != 0;
  };
  int bits = 0;
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    if (!nonzero(ld(q, 3 * sp + b)) && !nonzero(ld(q, 3 * cl + b))) continue;
#pragma unroll
    for (int a = 0; a < 3; ++a) bits |= nonzero(__ldg(u + (adj ? 3 * b + a : 3 * a + b))) ? 1 << a : 0;
  }
  return bits;
}

// Both hops of direction m added to acc in FP64, with the terms of the FP64
// kernels (SUM: the full operator's, which starts the backward product at the
// forward one and takes the difference from the two).  S: sign of the forward
// projector; m and S at run time, so that lanes with different m run together.
template <bool SUM, class Load>
__device__ __forceinline__ void fx_pair_f64(Load ld, const double2 *__restrict__ links, int m, int S, unsigned qf,
                                            unsigned s, unsigned qb, double2 (&acc)[12]) {
  // projection of 1 - gamma_m for the upper spins 0, 1 and reconstruction of 1 + gamma_m
  const int p0 = m == 3 ? 2 : m != 1, p1 = m == 0 ? 1 : m == 2 ? 3 : 2;
  const int r0 = m == 1 ? 2 : m != 3, r1 = m == 0 ? 1 : m == 2 ? 3 : 0;
  const int c0 = m < 2 ? 9 : 6, c1 = m < 2 ? 6 : 9;   // the lower spins that go with them
  double2 h[6], f[6], sum[6];
#pragma unroll
  for (int back = 0; back < 2; ++back) {
    const unsigned q = back ? qb : qf;
    const int flip = (back ? -S : S) > 0 ? 2 : 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      h[b] = cadd(ld(q, b), fx_turned(ld(q, c0 + b), (p0 + flip) & 3));
      h[3 + b] = cadd(ld(q, 3 + b), fx_turned(ld(q, c1 + b), (p1 + flip) & 3));
    }
    const double2 *u = links + ((size_t)(back ? qb : s) * 4 + m) * 9;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int sp = 0; sp < 2; ++sp) {
        double2 x = SUM && back ? f[3 * sp + a] : make_double2(0.0, 0.0);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          const double2 e = __ldg(u + (back ? 3 * b + a : 3 * a + b));
          x = back ? cfmac(e, h[3 * sp + b], x) : cfma(e, h[3 * sp + b], x);
        }
        (back ? sum : f)[3 * sp + a] = x;
      }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    double2 d[2];
#pragma unroll
    for (int sp = 0; sp < 2; ++sp) {
      const double2 cf = f[3 * sp + a], cb = sum[3 * sp + a];   // cb: with SUM the sum of both
      acc[3 * sp + a] = cadd(acc[3 * sp + a], SUM ? cb : cadd(cf, cb));
      d[sp] = SUM ? make_double2(fma(2.0, cf.x, -cb.x), fma(2.0, cf.y, -cb.y)) : csub(cf, cb);
    }
    const int flip = S > 0 ? 0 : 2;
    const double2 l0 = fx_turned(d[0], (r0 + flip) & 3), l1 = fx_turned(d[1], (r1 + flip) & 3);
    acc[6 + a] = cadd(acc[6 + a], m < 2 ? l1 : l0);
    acc[9 + a] = cadd(acc[9 + a], m < 2 ? l0 : l1);
  }
}

// FP64 hop sums of a warp's 16 sites for those that need them: special (values
// that fixed point does not hold), or lost components (fx_lost) with any nonzero
// term.  The whole warp calls it, a site's two lanes taking two directions each.
// Returns whether the site's sums were written to out.
template <bool DAG, bool SUM, class Load>
__device__ __forceinline__ bool fx_exact(Load ld, const double2 *__restrict__ links, const unsigned (&nup)[4],
                                         const unsigned (&ndn)[4], unsigned s, int sp, bool special, int lost,
                                         double2 *out) {
  constexpr int F = DAG ? +1 : -1;
  bool need = special;
  if (__any_sync(0xffffffffu, lost != 0 && !special)) {
    int up = 0, low = 0, xy = 0;
#pragma unroll 1
    for (int i = 0; i < 8; ++i) {
      const int m = i >> 1;
      const bool fwd = !(i & 1);
      const unsigned q = fwd ? nup[m] : ndn[m];
      const int t = fx_terms(ld, links + ((size_t)(fwd ? s : q) * 4 + m) * 9, !fwd, q, sp, m < 2 ? 3 - sp : 2 + sp);
      up |= t;
      if (m < 2) xy |= t;
      else low |= t;
    }
    low |= __shfl_xor_sync(0xffffffffu, xy, 16);
    need = need || (lost & (up | low << 3)) != 0;
  }
  need = __shfl_xor_sync(0xffffffffu, (int)need, 16) || need;
  if (!__any_sync(0xffffffffu, need)) return false;
  double2 acc[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) acc[c] = make_double2(0.0, 0.0);
#pragma unroll 1
  for (int i = 0; i < 2; ++i) {
    const int m = 2 * i + sp;
    fx_pair_f64<SUM>(ld, links, m, F, nup[m], s, ndn[m], acc);
  }
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    acc[c].x += __shfl_xor_sync(0xffffffffu, acc[c].x, 16);
    acc[c].y += __shfl_xor_sync(0xffffffffu, acc[c].y, 16);
    if (need && sp == c / 6) out[c] = acc[c];
  }
  return need;
}

// ----------------------------------------------------------------- a warp's entries

// Exponent field of an entry's larger part (at least FX_EMIN); ok becomes false
// where fixed point does not hold the entry.
__device__ __forceinline__ int fx_entry_exponent(double2 x, bool &ok) {
  const int e = max(exp_bits(x.x), exp_bits(x.y));
  const bool zero = ((__double_as_longlong(x.x) | __double_as_longlong(x.y)) << 1) == 0;
  ok = ok && (zero || (e >= FX_EMIN && e <= FX_EMAX));
  return max(e, FX_EMIN);
}

// Shared exponent of N entries a lane over the warp: the largest exponent field
// (FX_EMIN: all are zero) and, in ok, whether fixed point holds every value.
template <int N>
__device__ __forceinline__ int fx_warp_exponent(const double2 (&x)[N], bool &ok) {
  int e = 0;
  unsigned long long any = 0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    e = max(e, max(exp_bits(x[i].x), exp_bits(x[i].y)));
    any |= (unsigned long long)(__double_as_longlong(x[i].x) | __double_as_longlong(x[i].y)) << 1;
  }
  e = __reduce_max_sync(0xffffffffu, e);
  ok = e <= FX_EMAX && (e > FX_EMIN || !__any_sync(0xffffffffu, any != 0));
  return max(e, FX_EMIN);
}

// <a, v> and ||v||^2 over N <= 8 entries a lane of a warp, in fixed point
// against the warp's exponents: lane 0 returns (re, ||v||^2), lane 16 (im, ).
// A lane's sums are below 2^58 (middle 2^60), the warp's below 2^63; a product
// leaves out 2^-56 of the maxima's, a lane's sum is rounded at 2^-54.  That is below
// FP64's roundings unless the vectors have their large entries apart: a sum below
// 2^-5 of the maxima's product (2^48 units; one warp in 1e4 on even fields) is formed
// in FP64.  In FP64 this is six FMAs an entry, 76 clocks of a subpartition each
// for a warp, and as many for every addition of the warp's reduction.
template <int N>
__device__ __forceinline__ double2 fx_warp_dots(const double2 (&a)[N], const double2 (&v)[N]) {
  bool oka, okv;
  const int ea = fx_warp_exponent(a, oka), ev = fx_warp_exponent(v, okv);
  const bool upper = threadIdx.x & 16;
  if (oka && okv) {
    long long rh = 0, rm = 1LL << 29, ih = 0, im = 1LL << 29, nh = 0, nm = 1LL << 28;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int4 x = fx_cut30(a[i], ea), y = fx_cut30(v[i], ev);
      fx_wide(rh, x.x, y.x);
      fx_wide(rm, x.x, y.y);
      fx_wide(rm, x.y, y.x);
      fx_wide(rh, x.z, y.z);
      fx_wide(rm, x.z, y.w);
      fx_wide(rm, x.w, y.z);
      fx_wide(ih, x.x, y.z);
      fx_wide(im, x.x, y.w);
      fx_wide(im, x.y, y.z);
      fx_wide(ih, -x.z, y.x);
      fx_wide(im, -x.z, y.y);
      fx_wide(im, -x.w, y.x);
      fx_wide(nh, y.x, y.x);
      fx_wide(nm, y.x, y.y);
      fx_wide(nh, y.z, y.z);
      fx_wide(nm, y.z, y.w);
    }
    const long long tr = rh + (rm >> 30), ti = ih + (im >> 30);
    long long t = (upper ? ti : tr) + __shfl_xor_sync(0xffffffffu, upper ? tr : ti, 16);
    long long u = nh + (nm >> 29);
    u += __shfl_xor_sync(0xffffffffu, u, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      t += __shfl_xor_sync(0xffffffffu, t, o);
      u += __shfl_xor_sync(0xffffffffu, u, o);
    }
    const bool zero = ea == FX_EMIN || ev == FX_EMIN;
    if (zero || __any_sync(0xffffffffu, t >= 1LL << 48 || t <= -(1LL << 48)))
      return make_double2(fx_scaled(t, ea + ev - 1019), fx_scaled(u, ev + ev - 1019));
  }
  double s[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int i = 0; i < N; ++i) {
    s[0] = fma(a[i].x, v[i].x, fma(a[i].y, v[i].y, s[0]));
    s[1] = fma(a[i].x, v[i].y, fma(-a[i].y, v[i].x, s[1]));
    s[2] = fma(v[i].x, v[i].x, fma(v[i].y, v[i].y, s[2]));
  }
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
  return make_double2(upper ? s[1] : s[0], s[2]);
}

// Sum of the warps' fx_warp_dots over the block, written as its three
// partials <a, v> re, im and ||v||^2.  sh: WARPS entries.
template <int WARPS>
__device__ __forceinline__ void fx_block_dots(double2 d, double (*sh)[3], double *dst) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    sh[w][0] = d.x;
    sh[w][2] = d.y;
  } else if (lane == 16) {
    sh[w][1] = d.x;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < WARPS; ++i) s += sh[i][threadIdx.x];
    dst[threadIdx.x] = s;
  }
}

}  // namespace wd
