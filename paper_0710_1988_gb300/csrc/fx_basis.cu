// Krylov basis in block fixed point: the Gram-Schmidt products of GMRES-DR
// (Sec. 1), h = V^dagger w and w -= V h for one vector w.
//
// In FP64 both products are bound by the FP64 pipe (four FMAs, 2.4 clocks of
// an SM, for 16 bytes of V that memory delivers in 0.75).  As in fx.cuh the
// operands become integers: a vector is cut into chunks of FXB_CHUNK entries,
// each chunk shares the largest exponent field E of its entries and holds them as
// X = round(x 2^(1078 - E)) = hi 2^29 + lo, |hi| <= 2^27, |lo| <= 2^28, in
// two planes (hi: re, im; lo: re, im; 16 bytes an entry, as in FP64).  A real
// product is hi hi + (hi lo + lo hi) 2^-29, three 32 x 32 + 64-bit
// multiply-adds, twelve a complex product: 0.2 clocks of an SM at the 60 that a
// probe of independent chains issues, 0.4 at the 30 reached here, against 0.75 for
// the 16 bytes: both products then depend on memory first.
//
// Bounds.  Dot: a lane's four complex products are below 2^57 in the high sum
// and 2^60 in the middle one, a warp's sum of lanes below 2^62; the sums of
// warps and chunks are FP64.  Update: k <= 128 products are below 2^62 in the
// high sum; the middle sum, below 2^63 for 64 vectors, is folded in every 32.
// Error: a product leaves out lo lo, below 2^-56 of the chunk maxima's
// product, and a lane's sum is rounded at 2^-54 of it; FP64 rounds each
// partial sum (2^-53 of it, 2 k times an entry in the update).
//
// Chunks with infinities, NaN or magnitudes near the ends of FP64's range
// have exponent FX_SPECIAL and take their products in FP64.  So do results that
// rest on entries far below their chunk's largest, for which its unit is coarser
// than FP64's rounding: a warp's dot below 2^-5 of the maxima's product, and an
// entry of the update whose own value and partial sums all stay below 2^-6 of
// the largest |h_j| 2^(E_j).
#include "chain.cuh"
#include "cplx.cuh"
#include "fx.cuh"
#include "kernels.cuh"
#include "wd_internal.h"

namespace wd {

constexpr int FXB_THREADS = 192;
constexpr int FXB_CHUNK = 768;   // 64 sites of 12, four entries a thread
constexpr int FXB_JB = 16;       // most vectors of one dot block

long long fxb_chunks(long long n) { return (n + FXB_CHUNK - 1) / FXB_CHUNK; }

// A thread's four entries of a chunk: pairs 2 tid, 2 tid + 1 of both halves.
__device__ __forceinline__ int fxb_entry(int q) {
  return (q >> 1) * (FXB_CHUNK / 2) + 2 * (int)threadIdx.x + (q & 1);
}

__device__ __forceinline__ bool fxb_nonzero(double2 x) {
  return ((__double_as_longlong(x.x) | __double_as_longlong(x.y)) << 1) != 0;
}

// Largest exponent field over the block's entries and whether all are zero,
// as a shared exponent (fx_site_exponent); *raw the field itself.  red: two words a warp.
__device__ __forceinline__ int fxb_exponent(const double2 (&x)[4], int *raw, int *red) {
  int e = 0;
  unsigned long long any = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    e = max(e, max(exp_bits(x[q].x), exp_bits(x[q].y)));
    any |= (unsigned long long)(__double_as_longlong(x[q].x) | __double_as_longlong(x[q].y)) << 1;
  }
  e = __reduce_max_sync(0xffffffffu, e);
  const int nz = __any_sync(0xffffffffu, any != 0);
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    red[2 * w] = e;
    red[2 * w + 1] = nz;
  }
  __syncthreads();
  int m = 0, z = 0;
#pragma unroll
  for (int i = 0; i < FXB_THREADS / 32; ++i) {
    m = max(m, red[2 * i]);
    z |= red[2 * i + 1];
  }
  *raw = max(m, FX_EMIN);
  return fx_site_exponent(m, z == 0);
}

// ----------------------------------------------------------------- encoding

// v = w * (1 / H[idx].re) (H == nullptr: v = w) into the planes hi, lo and
// exponents ex of one or more vectors (blockIdx.y), with the FP64 values in v
// (unless nullptr or w itself) and, for the next operator product, the
// site-wise fixed point of fx.cuh (fx.v != nullptr; one vector).
__global__ void __launch_bounds__(FXB_THREADS)
fxb_encode_kernel(const double2 *w, const double2 *H, int idx, double2 *v, int2 *__restrict__ hi,
                  int2 *__restrict__ lo, int *__restrict__ ex, FxVec fx, long long n,
                  const int *status) {
  chain_enter();
  if (status != nullptr && *status != 0) return;
  __shared__ int red[2 * FXB_THREADS / 32];
  __shared__ int site_e[FXB_CHUNK / 12], site_nz[FXB_CHUNK / 12];
  __shared__ double s_inv;
  const long long j = blockIdx.y, base = (long long)blockIdx.x * FXB_CHUNK;
  if (H != nullptr && threadIdx.x == 0) s_inv = 1.0 / H[idx].x;   // one division a block
  if (fx.v != nullptr && threadIdx.x < FXB_CHUNK / 12) site_e[threadIdx.x] = site_nz[threadIdx.x] = 0;
  __syncthreads();
  double2 x[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const long long i = base + fxb_entry(q);
    x[q] = i < n ? w[j * n + i] : make_double2(0.0, 0.0);
    if (H != nullptr) x[q] = cscale(s_inv, x[q]);
    if (v != nullptr && i < n) v[j * n + i] = x[q];
    if (fx.v != nullptr) {
      const int s = fxb_entry(q) / 12;
      atomicMax(&site_e[s], max(exp_bits(x[q].x), exp_bits(x[q].y)));
      if ((__double_as_longlong(x[q].x) | __double_as_longlong(x[q].y)) << 1) site_nz[s] = 1;
    }
  }
  int raw;
  const int E = fxb_exponent(x, &raw, red);   // its barrier also orders the sites' exponents
  if (threadIdx.x == 0) ex[j * gridDim.x + blockIdx.x] = E;
#pragma unroll
  for (int q = 0; q < 4; q += 2) {
    const long long i = base + fxb_entry(q);
    if (i >= n) continue;   // n is even: a pair is inside or outside
    const int4 a = fx_slices(x[q], raw), b = fx_slices(x[q + 1], raw);
    *reinterpret_cast<int4 *>(hi + j * n + i) = make_int4(a.x, a.z, b.x, b.z);
    *reinterpret_cast<int4 *>(lo + j * n + i) = make_int4(a.y, a.w, b.y, b.w);
  }
  if (fx.v != nullptr) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = fxb_entry(q), s = c / 12;
      if (base + c >= n) continue;
      const unsigned site = (unsigned)((base + c) / 12);
      const int e = site_e[s];
      fx.v[fx_at(site, 12) + (c - 12 * s) * FX_TILE] = fx_slices(x[q], max(e, FX_EMIN));
      if (c == 12 * s) fx.e[site] = fx_site_exponent(e, site_nz[s] == 0);
    }
  }
}

cudaError_t launch_fxb_encode(const double2 *w, const double2 *H, int idx, double2 *v, FxBasis b,
                              long long j, int count, FxVec fx, long long n, const int *status,
                              cudaStream_t s) {
  ProfLaunch prof_(PC_STREAM, s);
  const long long nc = fxb_chunks(n);
  return launch_chained(fxb_encode_kernel, dim3((unsigned)nc, count), dim3(FXB_THREADS), 0, s, w, H, idx, v,
                        b.hi + j * n, b.lo + j * n, b.ex + j * nc, fx, n, status);
}

// ----------------------------------------------------------------- operands in flight

// A thread's entries of the next FXB_DEPTH vectors travel to shared memory
// while it works on one: 16-byte copies into its own slots, so no barrier and
// no registers (with the loads in registers the kernels wait for them: the
// dot 397 us where this form takes 116, 61 vectors on average at 16^4).
constexpr int FXB_DEPTH = 4;
struct FxbRing {
  int4 w[FXB_DEPTH][4][FXB_THREADS];   // hi and lo of both halves of the chunk
};

__device__ __forceinline__ void fxb_copy(int4 *dst, const int2 *src, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
               ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(in ? 16 : 0) : "memory");
}

// src: the thread's first entry in a plane (inside it even when in0 is false)
__device__ __forceinline__ void fxb_fetch(FxbRing &r, int slot, const int2 *hi, const int2 *lo, bool in0,
                                          bool in1) {
  const int t = threadIdx.x;
  fxb_copy(&r.w[slot][0][t], hi, in0);
  fxb_copy(&r.w[slot][1][t], lo, in0);
  fxb_copy(&r.w[slot][2][t], in1 ? hi + FXB_CHUNK / 2 : hi, in1);
  fxb_copy(&r.w[slot][3][t], in1 ? lo + FXB_CHUNK / 2 : lo, in1);
}

__device__ __forceinline__ void fxb_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void fxb_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// one real product: (ah, al) (bh, bl) into the high and middle sums
__device__ __forceinline__ void fxb_mac(long long &h, long long &m, int ah, int al, int bh, int bl) {
  fx_wide(h, ah, bh);
  fx_wide(m, ah, bl);
  fx_wide(m, al, bh);
}

// ----------------------------------------------------------------- dot

// Sum over the warp of two 64-bit values a lane: lanes 0 .. 15 get a's, 16 .. 31 b's.
__device__ __forceinline__ long long fxb_warp_sum(long long a, long long b) {
  const bool upper = threadIdx.x & 16;
  const long long send = upper ? a : b, keep = upper ? b : a;
  long long t = keep + __shfl_xor_sync(0xffffffffu, send, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// partial[(by gx + bx) jb + jj] = sum over the block's chunks of conj(V_j) w,
// j = by jb + jj < k; g5: w is gamma5 w.  A block encodes its chunk of w once
// for its jb <= 16 vectors and handles chunks bx, bx + gx, ...
__global__ void __launch_bounds__(FXB_THREADS, 3)
fxb_dot_kernel(FxBasis b, const double2 *V, int k, int jb, const double2 *W,
               int g5, long long n, double2 *__restrict__ partial, const int *status) {
  chain_enter();
  if (status != nullptr && *status != 0) return;
  extern __shared__ __align__(16) unsigned char fxb_smem[];
  FxbRing &ring = *reinterpret_cast<FxbRing *>(fxb_smem);
  __shared__ int red[2 * FXB_THREADS / 32];
  __shared__ long long tsum[FXB_THREADS / 32][2 * FXB_JB];
  __shared__ double wsum[FXB_THREADS / 32][2 * FXB_JB];
  const int j0 = blockIdx.y * jb, nj = min(jb, k - j0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long nc = (n + FXB_CHUNK - 1) / FXB_CHUNK;
  const int mine = 2 * (int)threadIdx.x;   // first entry of the thread in a chunk
  // the next operand to fetch: vector j0 + fj of chunk fc
  long long fc = blockIdx.x, fo = 0;   // fo: its first entry of this thread in the planes
  int fj = 0;
  bool in0 = false, in1 = false;
  auto fetch = [&](int slot) {
    if (fc < nc) {
      if (fj == 0) {
        const long long at = fc * FXB_CHUNK + mine;
        in0 = at < n;
        in1 = at + FXB_CHUNK / 2 < n;
        fo = (long long)j0 * n + (in0 ? at : 0);
      }
      fxb_fetch(ring, slot, b.hi + fo, b.lo + fo, in0, in1);
      fo += n;
      if (++fj == nj) fj = 0, fc += gridDim.x;
    }
    fxb_commit();
  };
#pragma unroll
  for (int u = 0; u < FXB_DEPTH - 1; ++u) fetch(u);
  int slot = 0;
  double sum = 0.0;   // lane l: value l (2 jj, 2 jj + 1: re, im of vector jj)
  for (long long c = blockIdx.x; c < nc; c += gridDim.x) {
    const long long base = c * FXB_CHUNK;
    double2 x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const long long i = base + fxb_entry(q);
      x[q] = i < n ? W[i] : make_double2(0.0, 0.0);
      if (g5 && fxb_entry(q) % 12 >= 6) x[q] = cneg(x[q]);
    }
    int raw;
    const int Ew = fxb_exponent(x, &raw, red);
    __syncthreads();   // red is reused by the next chunk
    int4 w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = fx_slices(x[q], raw);
    for (int jj = 0; jj < nj; ++jj) {
      fetch((slot + FXB_DEPTH - 1) % FXB_DEPTH);
      fxb_wait<FXB_DEPTH - 1>();
      long long rh = 0, rm = 1LL << 28, ih = 0, im = 1LL << 28;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int4 h = ring.w[slot][2 * half][threadIdx.x], l = ring.w[slot][2 * half + 1][threadIdx.x];
#pragma unroll
        for (int o = 0; o < 2; ++o) {
          const int4 y = w[2 * half + o];
          const int ah = o ? h.z : h.x, al = o ? l.z : l.x;   // re
          const int bh = o ? h.w : h.y, bl = o ? l.w : l.y;   // im
          fxb_mac(rh, rm, ah, al, y.x, y.y);
          fxb_mac(rh, rm, bh, bl, y.z, y.w);
          fxb_mac(ih, im, ah, al, y.z, y.w);
          fxb_mac(ih, im, -bh, -bl, y.x, y.y);
        }
      }
      const long long T = fxb_warp_sum(rh + (rm >> 29), ih + (im >> 29));
      if ((lane & 15) == 0) tsum[warp][2 * jj + (lane >> 4)] = T;
      slot = (slot + 1) % FXB_DEPTH;
    }
    __syncwarp();
    const int jl = lane >> 1;   // this lane's vector
    const int Ev = jl < nj ? b.ex[(long long)(j0 + jl) * nc + c] : 0;
    const long long T = jl < nj ? tsum[warp][lane] : 0;
    // long enough (2^47 units; one in 1e4 is not on even fields), or a chunk of zeros
    const bool mine_long = T >= 1LL << 47 || T <= -(1LL << 47) || Ev == 0 || Ew == 0;
    const bool longer = __shfl_xor_sync(0xffffffffu, (int)mine_long, 1) || mine_long;
    const bool held = Ew != FX_SPECIAL && Ev != FX_SPECIAL && longer;
    if (jl < nj && held) sum += fx_scaled(T, Ev + Ew - 1019);
    const unsigned other = __ballot_sync(0xffffffffu, jl < nj && !held);
    const unsigned spec = __ballot_sync(0xffffffffu, Ew == FX_SPECIAL || Ev == FX_SPECIAL);
    // the others in FP64
    for (int jj = 0; other != 0 && jj < nj; ++jj) {
      if (!((other >> (2 * jj)) & 1u)) continue;
      const long long j = j0 + jj;
      double2 a = make_double2(0.0, 0.0), v[4];
      bool terms = (spec >> (2 * jj)) & 1u;   // infinities times zero count
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long long i = base + fxb_entry(q);
        v[q] = i < n ? V[j * n + i] : make_double2(0.0, 0.0);
        terms = terms || (fxb_nonzero(v[q]) && fxb_nonzero(x[q]));
      }
      if (!__any_sync(0xffffffffu, terms)) continue;   // as in regions that a source has not reached
#pragma unroll
      for (int q = 0; q < 4; ++q) a = cfmac(v[q], x[q], a);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
        a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
      }
      if (jl == jj) sum += lane & 1 ? a.y : a.x;
    }
  }
  fxb_wait<0>();
  wsum[warp][lane] = sum;
  __syncthreads();
  if ((int)threadIdx.x < nj) {
    const int q = threadIdx.x;
    double2 a = make_double2(0.0, 0.0);
#pragma unroll
    for (int i = 0; i < FXB_THREADS / 32; ++i) {
      a.x += wsum[i][2 * q];
      a.y += wsum[i][2 * q + 1];
    }
    partial[((long long)blockIdx.y * gridDim.x + blockIdx.x) * jb + q] = a;
  }
}

// shared memory above 48 KB, once per device and thread
static cudaError_t fxb_allow_smem(const void *kernel, int *device) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev == *device) return e;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(FxbRing));
  if (e == cudaSuccess) *device = dev;
  return e;
}

// Grid: vectors in groups of at most 16, chunks over three blocks per
// SM in equal shares.
static void fxb_dot_grid(long long n, int k, dim3 *grid, int *jb) {
  const int gy = (k + FXB_JB - 1) / FXB_JB;
  const long long nc = fxb_chunks(n);
  long long gx = 456 / gy;
  if (gx < 1) gx = 1;
  if (gx > nc) gx = nc;
  const long long each = (nc + gx - 1) / gx;
  gx = (nc + each - 1) / each;
  *grid = dim3((unsigned)gx, gy);
  *jb = (k + gy - 1) / gy;
}

size_t fxb_dot_partials(long long n, int k) {
  dim3 g;
  int jb;
  fxb_dot_grid(n, k, &g, &jb);
  return (size_t)g.x * g.y * jb;
}

// C[j ldc] = conj(V_j) w (g5: conj(V_j) gamma5 w), C2[j ldc2] += the same
cudaError_t launch_fxb_dot(FxBasis b, const double2 *V, int k, const double2 *w, int g5, long long n,
                           double2 *partial, double2 *C, int ldc, double2 *C2, int ldc2,
                           const int *status, cudaStream_t s) {
  ProfLaunch prof_(PC_TS, s);
  if (k < 1) return cudaErrorInvalidValue;
  dim3 grid;
  int jb;
  fxb_dot_grid(n, k, &grid, &jb);
  static thread_local int device = -1;
  cudaError_t e = fxb_allow_smem((const void *)fxb_dot_kernel, &device);
  if (e != cudaSuccess) return e;
  e = launch_chained(fxb_dot_kernel, grid, dim3(FXB_THREADS), sizeof(FxbRing), s, b, V, k, jb, w, g5, n, partial, status);
  if (e != cudaSuccess) return e;
  return launch_ts_dot_finalize_grid(partial, (int)grid.x, (int)grid.y, jb, 1, k, 1, C, ldc, C2, ldc2, status, s);
}

// ----------------------------------------------------------------- update

// w -= V h (add: w += V h) for k vectors: a block's chunk of w in FP64, the
// sum V h in fixed point against the largest |h_j| 2^(E_j) of the chunk.
__global__ void __launch_bounds__(FXB_THREADS, 3)
fxb_update_kernel(FxBasis b, const double2 *V, int k, const double2 *h, int ldh,
                  int add, double2 *w, long long n, const int *status) {
  chain_enter();
  if (status != nullptr && *status != 0) return;
  __shared__ int4 g[128];       // h_j in slices
  __shared__ int top[FXB_THREADS / 32], bad[FXB_THREADS / 32];
  const long long c = blockIdx.x, nc = gridDim.x, base = c * FXB_CHUNK;
  const long long at = base + 2 * (int)threadIdx.x;
  const bool in0 = at < n, in1 = at + FXB_CHUNK / 2 < n;
  // exponent field of max(|re|, |im|) of h_j, plus E_j: the chunk's largest is G
  double2 hj = make_double2(0.0, 0.0);
  int ej = 0, Ej = 0;
  bool special = false;
  if ((int)threadIdx.x < k) {
    hj = h[(long long)threadIdx.x * ldh];
    Ej = b.ex[(long long)threadIdx.x * nc + c];
    ej = max(exp_bits(hj.x), exp_bits(hj.y));
    const bool zero = ((__double_as_longlong(hj.x) | __double_as_longlong(hj.y)) << 1) == 0;
    special = Ej == FX_SPECIAL || fx_site_exponent(ej, zero) == FX_SPECIAL;
  }
  const int mine = Ej != 0 && ej != 0 && !special ? Ej + ej : 0;
  const int wm = __reduce_max_sync(0xffffffffu, mine);
  const int wb = __any_sync(0xffffffffu, special);
  if ((threadIdx.x & 31) == 0) {
    top[threadIdx.x >> 5] = wm;
    bad[threadIdx.x >> 5] = wb;
  }
  __syncthreads();
  int G = 0, any_bad = 0;
#pragma unroll
  for (int i = 0; i < FXB_THREADS / 32; ++i) {
    G = max(G, top[i]);
    any_bad |= bad[i];
  }
  if ((int)threadIdx.x < k) g[threadIdx.x] = mine ? fx_slices(hj, G - Ej) : make_int4(0, 0, 0, 0);
  __syncthreads();
  if (any_bad) {   // in FP64
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const long long i = base + fxb_entry(q);
      if (i >= n) continue;
      double2 acc = make_double2(0.0, 0.0);
      for (int j = 0; j < k; ++j) acc = cfma(V[(long long)j * n + i], h[(long long)j * ldh], acc);
      w[i] = add ? cadd(w[i], acc) : csub(w[i], acc);
    }
    return;
  }
  extern __shared__ __align__(16) unsigned char fxb_smem[];
  FxbRing &ring = *reinterpret_cast<FxbRing *>(fxb_smem);
  auto fetch = [&](int slot, int j) {
    const long long o = (long long)j * n + (in0 ? at : 0);
    if (j < k) fxb_fetch(ring, slot, b.hi + o, b.lo + o, in0, in1);
    fxb_commit();
  };
#pragma unroll
  for (int u = 0; u < FXB_DEPTH - 1; ++u) fetch(u, u);
  double2 x[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) x[q] = (q < 2 ? in0 : in1) ? w[base + fxb_entry(q)] : make_double2(0.0, 0.0);
  long long rh[4], rm[4], ih[4], im[4];
  int reach[4];   // high words of the partial sums, or-ed; 2^47 units where x is large enough itself
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    rh[q] = ih[q] = 0;
    reach[q] = max(exp_bits(x[q].x), exp_bits(x[q].y)) >= G - 1028 ? 1 << 15 : 0;
  }
  auto track = [&]() {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int a = (int)(rh[q] >> 32), c2 = (int)(ih[q] >> 32);
      reach[q] |= (a ^ (a >> 31)) | (c2 ^ (c2 >> 31));
    }
  };
  for (int j0 = 0; j0 < k; j0 += 32) {
#pragma unroll
    for (int q = 0; q < 4; ++q) rm[q] = im[q] = 1LL << 28;
    const int j1 = min(k, j0 + 32);
    for (int j = j0; j < j1; ++j) {
      fetch((j + FXB_DEPTH - 1) % FXB_DEPTH, j + FXB_DEPTH - 1);
      fxb_wait<FXB_DEPTH - 1>();
      const int4 y = g[j];
      const int slot = j % FXB_DEPTH;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int4 hh = ring.w[slot][2 * (q >> 1)][threadIdx.x], l = ring.w[slot][2 * (q >> 1) + 1][threadIdx.x];
        const int ah = q & 1 ? hh.z : hh.x, al = q & 1 ? l.z : l.x;   // re
        const int bh = q & 1 ? hh.w : hh.y, bl = q & 1 ? l.w : l.y;   // im
        fxb_mac(rh[q], rm[q], ah, al, y.x, y.y);
        fxb_mac(rh[q], rm[q], -bh, -bl, y.z, y.w);
        fxb_mac(ih[q], im[q], ah, al, y.z, y.w);
        fxb_mac(ih[q], im[q], bh, bl, y.x, y.y);
      }
      if ((j & 3) == 3) track();
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      rh[q] += rm[q] >> 29;
      ih[q] += im[q] >> 29;
    }
  }
  track();
  // units 2^(58 - 2 * 1078 + G)
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (!(q < 2 ? in0 : in1)) continue;
    double re = fx_scaled(rh[q], G - 1019), im2 = fx_scaled(ih[q], G - 1019);
    if (reach[q] < 1 << 15 && G != 0) {   // G = 0: all products are zero
      double2 acc = make_double2(0.0, 0.0);
      for (int j = 0; j < k; ++j) {
        const double2 v = V[(long long)j * n + base + fxb_entry(q)];
        if (fxb_nonzero(v)) acc = cfma(v, h[(long long)j * ldh], acc);
      }
      re = acc.x;
      im2 = acc.y;
    }
    if (add) {
      re = -re;
      im2 = -im2;
    }
    w[base + fxb_entry(q)] = make_double2(x[q].x - re, x[q].y - im2);
  }
}

cudaError_t launch_fxb_update(FxBasis b, const double2 *V, int k, const double2 *h, int ldh, int add,
                              double2 *w, long long n, const int *status, cudaStream_t s) {
  ProfLaunch prof_(PC_TS, s);
  if (k < 1 || k > 128) return cudaErrorInvalidValue;
  static thread_local int device = -1;
  cudaError_t e = fxb_allow_smem((const void *)fxb_update_kernel, &device);
  if (e != cudaSuccess) return e;
  return launch_chained(fxb_update_kernel, dim3((unsigned)fxb_chunks(n)), dim3(FXB_THREADS), sizeof(FxbRing), s, b,
                        V, k, h, ldh, add, w, n, status);
}

// ----------------------------------------------------------------- correction

// w -= V h for the second pass of classical Gram-Schmidt and the block's
// partial of ||w||^2 afterwards.  The coefficients h are of the order of the
// first pass's rounding (|h| ~ eps ||w||): the correction V h then needs only
// FP32 accuracy relative to itself, far below FP64 rounding of w, and reads
// only the high plane (half the bytes of V; entries that are below 2^-4 of their
// chunk's largest in every vector are read from V).  FP32 path, taken when ||h||^2 <=
// 1e-20 (||w0||^2 - ||hsum||^2) (the correction below 1e-10 of the vector it
// corrects; ||w0||^2 from the Wilson kernel's partials, hsum the coefficients
// of both passes); products and sums in FP32, w updated in FP64.  Otherwise,
// and for chunks with FX_SPECIAL, FP64.  Every block forms the decision from
// the same device data in the same order, so all take the same path.
__global__ void __launch_bounds__(FXB_THREADS)
fxb_correction_kernel(FxBasis b, const double2 *V, int k, const double2 *h,
                      const double2 *hsum, int ldh, const double *part_w,
                      int nbw, double2 *w, long long n, double *__restrict__ part_n,
                      const int *status) {
  chain_enter();
  if (status != nullptr && *status != 0) return;
  __shared__ float2 hf[128];
  __shared__ int use32, bad;
  const long long c = blockIdx.x, nc = gridDim.x, base = c * FXB_CHUNK;
  if (threadIdx.x == 0) bad = 0;
  if (threadIdx.x < 32) {
    double w2 = 0.0, s2 = 0.0, c2 = 0.0;
    for (int i = threadIdx.x; i < nbw; i += 32) w2 += part_w[(long long)i * 3 + 2];
    for (int r = threadIdx.x; r < k; r += 32) {
      c2 += cnorm2(h[r]);
      s2 += cnorm2(hsum[(long long)r * ldh]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      w2 += __shfl_xor_sync(0xffffffffu, w2, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
      c2 += __shfl_xor_sync(0xffffffffu, c2, o);
    }
    if (threadIdx.x == 0) use32 = c2 <= 1e-20 * (w2 - s2) ? 1 : 0;
  }
  __syncthreads();
  if ((int)threadIdx.x < k) {
    const int E = b.ex[(long long)threadIdx.x * nc + c];
    if (E == FX_SPECIAL) bad = 1;
    const double2 hj = h[threadIdx.x];   // times the value of one unit of the high plane
    hf[threadIdx.x] = make_float2((float)ldexp(hj.x, E - 1049), (float)ldexp(hj.y, E - 1049));
  }
  __syncthreads();
  const bool fp32 = use32 != 0 && bad == 0;
  const long long at = base + 2 * (int)threadIdx.x;
  double red[1] = {0.0};
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const long long i = at + half * (FXB_CHUNK / 2);
    if (i >= n) continue;
    double2 o0 = w[i], o1 = w[i + 1];
    if (fp32) {
      float ax = 0.f, ay = 0.f, bx = 0.f, by = 0.f, am = 0.f, bm = 0.f;
#pragma unroll 8
      for (int r = 0; r < k; ++r) {
        const int4 v = *reinterpret_cast<const int4 *>(b.hi + (long long)r * n + i);
        const float2 y = hf[r];
        const float p = (float)v.x, q = (float)v.y, s = (float)v.z, t = (float)v.w;
        am = fmaxf(am, fmaxf(fabsf(p), fabsf(q)));
        bm = fmaxf(bm, fmaxf(fabsf(s), fabsf(t)));
        ax = fmaf(p, y.x, fmaf(-q, y.y, ax));
        ay = fmaf(p, y.y, fmaf(q, y.x, ay));
        bx = fmaf(s, y.x, fmaf(-t, y.y, bx));
        by = fmaf(s, y.y, fmaf(t, y.x, by));
      }
      // entries whose high parts have fewer than FP32's 24 bits in every vector: from V
      for (int one = 0; one < 2; ++one) {
        if ((one ? bm : am) >= 0x1p23f) continue;
        float2 c2 = make_float2(0.f, 0.f);
        for (int r = 0; r < k; ++r) {
          const double2 v = V[(long long)r * n + i + one];
          if (!fxb_nonzero(v)) continue;
          const int E = b.ex[(long long)r * nc + c];
          const float p = (float)ldexp(v.x, 1049 - E), q = (float)ldexp(v.y, 1049 - E);
          c2.x = fmaf(p, hf[r].x, fmaf(-q, hf[r].y, c2.x));
          c2.y = fmaf(p, hf[r].y, fmaf(q, hf[r].x, c2.y));
        }
        if (one) bx = c2.x, by = c2.y;
        else ax = c2.x, ay = c2.y;
      }
      o0 = make_double2(o0.x - (double)ax, o0.y - (double)ay);
      o1 = make_double2(o1.x - (double)bx, o1.y - (double)by);
    } else {
      double2 a0 = make_double2(0.0, 0.0), a1 = a0;
      for (int r = 0; r < k; ++r) {
        a0 = cfma(V[(long long)r * n + i], h[r], a0);
        a1 = cfma(V[(long long)r * n + i + 1], h[r], a1);
      }
      o0 = csub(o0, a0);
      o1 = csub(o1, a1);
    }
    w[i] = o0;
    w[i + 1] = o1;
    red[0] = fma(o0.x, o0.x, red[0]);
    red[0] = fma(o0.y, o0.y, red[0]);
    red[0] = fma(o1.x, o1.x, red[0]);
    red[0] = fma(o1.y, o1.y, red[0]);
  }
  block_sum<1>(red);
  if (threadIdx.x == 0) part_n[2 * c] = red[0];   // stride 2, as norms_kernel's
}

cudaError_t launch_fxb_correction(FxBasis b, const double2 *V, int k, const double2 *h,
                                  const double2 *hsum, int ldh, const double *part_w, int nbw,
                                  double2 *w, long long n, double *part_n, const int *status,
                                  cudaStream_t s) {
  ProfLaunch prof_(PC_TS, s);
  if (k < 1 || k > 128) return cudaErrorInvalidValue;
  return launch_chained(fxb_correction_kernel, dim3((unsigned)fxb_chunks(n)), dim3(FXB_THREADS), 0, s, b, V, k, h,
                        hsum, ldh, part_w, nbw, w, n, part_n, status);
}

}  // namespace wd
