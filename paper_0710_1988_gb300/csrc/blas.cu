// Streaming vector kernels of BiCGStab and GMRES-DR (FP64), their scalar
// finalizers, and the tall-skinny products V^dagger W and W += V Y.
//
// Every kernel is batched over right-hand sides (blockIdx.y = system) and
// skips systems whose status is not in its mask.  Reductions are
// deterministic: a fixed number of blocks per system, each block reduces
// in a fixed shuffle/shared-memory order and writes one partial, and a
// finalizer sums the partials in block order.
#include <cstdio>

#include "bicg_fin.cuh"
#include "chain.cuh"
#include "cplx.cuh"
#include "kernels.cuh"
#include "wd_internal.h"

namespace wd {

constexpr int SB_THREADS = 256;

int stream_blocks(long long n) {
  long long b = (n + SB_THREADS * 4 - 1) / (SB_THREADS * 4);
  if (b > 608) b = 608;  // 4 blocks per SM on 152 SMs
  if (b < 1) b = 1;
  return (int)b;
}

__device__ __forceinline__ bool sys_on(const int *status, unsigned mask, int r) {
  return status == nullptr || ((mask >> status[r]) & 1u);
}

// ----------------------------------------------------------------- vectors and norms

__global__ void __launch_bounds__(SB_THREADS)
sub_norm_kernel(double2 *__restrict__ out, const double2 *__restrict__ a,
                const double2 *__restrict__ b, const int *__restrict__ status, unsigned mask,
                double *__restrict__ partial, long long n) {
  const int r = blockIdx.y;
  if (!sys_on(status, mask, r)) return;
  const long long off = (long long)r * n;
  double red[1] = {0.0};
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const double2 v = csub(a[off + i], b[off + i]);
    out[off + i] = v;
    red[0] = fma(v.x, v.x, red[0]);
    red[0] = fma(v.y, v.y, red[0]);
  }
  block_sum<1>(red);
  if (threadIdx.x == 0) partial[(long long)r * gridDim.x + blockIdx.x] = red[0];
}

__global__ void __launch_bounds__(SB_THREADS)
norms_kernel(const double2 *__restrict__ a, const double2 *__restrict__ b,
             double *__restrict__ partial, long long n) {
  const int r = blockIdx.y;
  const long long off = (long long)r * n;
  double red[2] = {0.0, 0.0};
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const double2 v = a[off + i];
    red[0] = fma(v.x, v.x, red[0]);
    red[0] = fma(v.y, v.y, red[0]);
    if (b != nullptr) {
      const double2 w = b[off + i];
      red[1] = fma(w.x, w.x, red[1]);
      red[1] = fma(w.y, w.y, red[1]);
    }
  }
  block_sum<2>(red);
  if (threadIdx.x == 0) {
    double *d = partial + ((long long)r * gridDim.x + blockIdx.x) * 2;
    d[0] = red[0];
    d[1] = red[1];
  }
}

__global__ void __launch_bounds__(SB_THREADS)
restart_vectors_kernel(double2 *__restrict__ rhat, const double2 *__restrict__ rv,
                       double2 *__restrict__ p, double2 *__restrict__ v,
                       const int *__restrict__ status, unsigned mask, long long n) {
  const int r = blockIdx.y;
  if (!sys_on(status, mask, r)) return;
  const long long off = (long long)r * n;
  const double2 z = make_double2(0.0, 0.0);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    rhat[off + i] = rv[off + i];
    p[off + i] = z;
    v[off + i] = z;
  }
}

cudaError_t launch_sub_norm(double2 *out, const double2 *a, const double2 *b, const int *status,
                            unsigned mask, double *partial, long long n, int nrhs,
                            cudaStream_t s) {
  ProfLaunch prof_(PC_STREAM, s);
  sub_norm_kernel<<<dim3(stream_blocks(n), nrhs), SB_THREADS, 0, s>>>(out, a, b, status, mask,
                                                                      partial, n);
  return cudaGetLastError();
}
cudaError_t launch_norms(const double2 *a, const double2 *b, double *partial, long long n,
                         int nrhs, cudaStream_t s) {
  ProfLaunch prof_(PC_STREAM, s);
  norms_kernel<<<dim3(stream_blocks(n), nrhs), SB_THREADS, 0, s>>>(a, b, partial, n);
  return cudaGetLastError();
}
cudaError_t launch_bicg_restart_vectors(double2 *rhat, const double2 *r, double2 *p,
                                        double2 *v, const int *status, unsigned mask,
                                        long long n, int nrhs, cudaStream_t s) {
  ProfLaunch prof_(PC_STREAM, s);
  restart_vectors_kernel<<<dim3(stream_blocks(n), nrhs), SB_THREADS, 0, s>>>(rhat, r, p, v,
                                                                             status, mask, n);
  return cudaGetLastError();
}

// ----------------------------------------------------------------- finalizers

template <int NQ>
__device__ void reduce_partials(const double *partial, int nb, int r, double (&v)[NQ]) {
#pragma unroll
  for (int q = 0; q < NQ; ++q) v[q] = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const double *src = partial + ((long long)r * nb + b) * NQ;
#pragma unroll
    for (int q = 0; q < NQ; ++q) v[q] += src[q];
  }
  block_sum<NQ>(v);
}

// One block per system.
__global__ void __launch_bounds__(1024)
bicg_finalize_kernel(int kind, const double *partial, int nb, BicgScalars *sc,
                     int *status, double *hist, int hist_len) {
  chain_enter();
  const int r = blockIdx.x;
  const int st = status[r];
  if (kind == FIN_INIT) {  // partial: ||b||^2, ||r0||^2 (NQ = 2)
    double v[2];
    reduce_partials<2>(partial, nb, r, v);
    if (threadIdx.x == 0) {
      BicgScalars &S = sc[r];
      S.bnorm = sqrt(v[0]);
      const double rr = v[1];
      reset_recurrence(S, rr);
      if (S.bnorm == 0.0) {
        S.true_rel = 0.0;
        status[r] = ST_DONE;
      } else if (S.rnorm / S.bnorm <= S.tol) {
        status[r] = ST_RECURSIVE;
      } else {
        status[r] = ST_RESTART;
      }
    }
    return;
  }
  if (kind == FIN_ALPHA || kind == FIN_OMEGA || kind == FIN_RHO) {
    if (st != ST_ACTIVE) return;
    fin_system(kind, partial, nb, sc, status, hist, hist_len, r);
    return;
  }
  if (kind == FIN_TRUE) {  // ||b - A x||^2 (NQ = 1)
    if (st != ST_RECURSIVE && st != ST_BREAKDOWN && st != ST_MAXITER) return;
    double v[1];
    reduce_partials<1>(partial, nb, r, v);
    if (threadIdx.x != 0) return;
    BicgScalars &S = sc[r];
    S.mvp_extra += 1;
    S.true_rel = sqrt(v[0]) / S.bnorm;
    if (st != ST_RECURSIVE) return;  // final anyway; just record
    if (S.true_rel <= S.tol) {
      status[r] = ST_DONE;
    } else if (S.restarts < S.max_restarts) {
      S.restarts += 1;
      reset_recurrence(S, v[0]);
      status[r] = ST_RESTART;
    } else {
      status[r] = ST_FAILED;
    }
    return;
  }
  // FIN_ACTIVATE: restart vectors are in place
  if (threadIdx.x == 0 && st == ST_RESTART) status[r] = ST_ACTIVE;
}

cudaError_t launch_bicg_finalize(int kind, const double *partial, int nb, BicgScalars *sc,
                                 int *status, double *hist, int hist_len, int nrhs,
                                 cudaStream_t s) {
  ProfLaunch prof_(PC_STREAM, s);
  return launch_chained(bicg_finalize_kernel, dim3(nrhs), dim3(nb > 1024 ? 1024 : 256), 0, s, kind, partial, nb, sc, status, hist, hist_len);
}

// ----------------------------------------------------------------- tall-skinny
//
// Both products are FP64-ALU bound on this part (4 DFMA per complex
// element pair against ~0.3 DFMA/byte of machine balance), so the kernels
// are shaped to issue nothing but the DFMAs the product needs: every thread
// walks vector elements, keeps a JT x RT (dot) or NC (update) tile of
// complex accumulators in registers, and the block reduces once at the end.

constexpr int TS_THREADS = 256;

static void ts_dot_tile(int nrhs, int *JT, int *RT) {
  *RT = nrhs >= 2 ? 2 : 1;
  *JT = *RT == 1 ? 16 : 8;
}

static void ts_dot_grid(long long n, int k, int nrhs, dim3 *grid) {
  int JT, RT;
  ts_dot_tile(nrhs, &JT, &RT);
  const int gy = (k + JT - 1) / JT, gz = (nrhs + RT - 1) / RT;
  long long gx = TS_MAX_BLOCKS / (gy * gz);
  const long long need = (n + TS_THREADS - 1) / TS_THREADS;
  if (gx > need) gx = need;
  if (gx < 8) gx = need < 8 ? need : 8;
  if (gx < 1) gx = 1;
  *grid = dim3((unsigned)gx, gy, gz);
}

int ts_dot_blocks(long long n, int k, int nrhs) {
  dim3 g;
  ts_dot_grid(n, k, nrhs, &g);
  return (int)(g.x * g.y * g.z);
}

// Block reduction of a tile of 16 complex sums (32 doubles per thread) in a
// fixed order, written as the block's partials.  Within a warp the 32
// doubles are reduced by recursive halving: at each of the five levels a
// lane keeps half of its values, sends the other half to its partner and
// adds what it receives, so lane i ends with the warp sum of value i after
// 16 + 8 + 4 + 2 + 1 additions (a shuffle tree per value would take 160).
__device__ __forceinline__ void ts_tile_reduce(double (&vals)[32], double2 *__restrict__ partial) {
  __shared__ double red[32][TS_THREADS / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int lvl = 0; lvl < 5; ++lvl) {
    const int half = 16 >> lvl;           // values kept after this level
    const bool upper = (lane >> (4 - lvl)) & 1;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const double send = upper ? vals[i] : vals[i + half];
      const double keep = upper ? vals[i + half] : vals[i];
      vals[i] = keep + __shfl_xor_sync(0xffffffffu, send, half);
    }
  }
  red[lane][wid] = vals[0];
  __syncthreads();
  const long long tile = ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  for (int q = threadIdx.x; q < 16; q += blockDim.x) {
    double a = 0.0, b = 0.0;
    for (int w2 = 0; w2 < TS_THREADS / 32; ++w2) {
      a += red[q * 2][w2];
      b += red[q * 2 + 1][w2];
    }
    partial[tile * 16 + q] = make_double2(a, b);
  }
}

template <int JT, int RT>
__global__ void __launch_bounds__(TS_THREADS)
ts_dot_kernel(const double2 *__restrict__ V, int k, const double2 *__restrict__ W, int nrhs,
              int g5, long long n, double2 *__restrict__ partial,
              const int *__restrict__ status) {
  if (status != nullptr && *status != 0) return;
  const int j0 = blockIdx.y * JT, r0 = blockIdx.z * RT;
  const int nj = min(JT, k - j0), nr = min(RT, nrhs - r0);
  double2 acc[JT][RT];
#pragma unroll
  for (int j = 0; j < JT; ++j)
#pragma unroll
    for (int r = 0; r < RT; ++r) acc[j][r] = make_double2(0.0, 0.0);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    double2 w[RT];
    const bool neg = g5 && (i % 12) >= 6;  // gamma5 = diag(1, 1, -1, -1)
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      w[r] = r < nr ? __ldg(W + (long long)(r0 + r) * n + i) : make_double2(0.0, 0.0);
      if (neg) w[r] = cneg(w[r]);
    }
#pragma unroll
    for (int j = 0; j < JT; ++j) {
      if (j < nj) {
        const double2 v = __ldg(V + (long long)(j0 + j) * n + i);
#pragma unroll
        for (int r = 0; r < RT; ++r) acc[j][r] = cfmac(v, w[r], acc[j][r]);
      }
    }
  }
  double vals[32];
#pragma unroll
  for (int j = 0; j < JT; ++j)
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      vals[(j * RT + r) * 2] = acc[j][r].x;
      vals[(j * RT + r) * 2 + 1] = acc[j][r].y;
    }
  static_assert(JT * RT * 2 == 32, "the tile holds 32 doubles");
  ts_tile_reduce(vals, partial);
}

// One warp per (j, r) pair: the lanes load the gx block partials of the pair
// together (lane b, b + 32, ...) and reduce them with a fixed shuffle tree,
// so the loads overlap instead of forming one dependent chain.
__global__ void ts_dot_finalize_kernel(const double2 *partial, int gx, int gy,
                                       int JT, int RT, int k, int nrhs, double2 *C, int ldc,
                                       double2 *C2, int ldc2, const int *status) {
  chain_enter();
  if (status != nullptr && *status != 0) return;
  const int P = k * nrhs;
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  for (int pair = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; pair < P; pair += warps) {
    const int j = pair / nrhs, r = pair % nrhs;
    const int ty = j / JT, jj = j % JT, tz = r / RT, rr = r % RT;
    const long long base = ((long long)tz * gy + ty) * gx;
    double2 t = make_double2(0.0, 0.0);
    for (int b = lane; b < gx; b += 32) t = cadd(t, partial[(base + b) * JT * RT + jj * RT + rr]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      t.x += __shfl_xor_sync(0xffffffffu, t.x, off);
      t.y += __shfl_xor_sync(0xffffffffu, t.y, off);
    }
    if (lane == 0) {
      C[(long long)j * ldc + r] = t;
      if (C2 != nullptr) {
        double2 &d = C2[(long long)j * ldc2 + r];
        d = cadd(d, t);
      }
    }
  }
}

cudaError_t launch_ts_dot(const double2 *V, int k, const double2 *W, int nrhs, int g5,
                          long long n, double2 *partial, const int *status, cudaStream_t s) {
  ProfLaunch prof_(PC_TS, s);
  if (k < 1 || nrhs < 1 || k > 4096 || nrhs > 4096) return cudaErrorInvalidValue;
  dim3 grid;
  ts_dot_grid(n, k, nrhs, &grid);
  int JT, RT;
  ts_dot_tile(nrhs, &JT, &RT);
  if (RT == 1)
    ts_dot_kernel<16, 1><<<grid, TS_THREADS, 0, s>>>(V, k, W, nrhs, g5, n, partial, status);
  else
    ts_dot_kernel<8, 2><<<grid, TS_THREADS, 0, s>>>(V, k, W, nrhs, g5, n, partial, status);
  return cudaGetLastError();
}

cudaError_t launch_ts_dot_finalize_grid(const double2 *partial, int gx, int gy, int JT, int RT, int k,
                                        int nrhs, double2 *C, int ldc, double2 *C2, int ldc2,
                                        const int *status, cudaStream_t s) {
  const int P = k * nrhs;  // one warp per pair, four warps per block
  return launch_chained(ts_dot_finalize_kernel, dim3((P + 3) / 4), dim3(128), 0, s, partial, gx, gy, JT, RT, k, nrhs,
                        C, ldc, C2, ldc2, status);
}

cudaError_t launch_ts_dot_finalize(const double2 *partial, long long n, int k, int nrhs,
                                   double2 *C, int ldc, double2 *C2, int ldc2,
                                   const int *status, cudaStream_t s) {
  ProfLaunch prof_(PC_TS, s);
  dim3 grid;
  ts_dot_grid(n, k, nrhs, &grid);
  int JT, RT;
  ts_dot_tile(nrhs, &JT, &RT);
  return launch_ts_dot_finalize_grid(partial, (int)grid.x, (int)grid.y, JT, RT, k, nrhs, C, ldc, C2, ldc2,
                                     status, s);
}

constexpr int TU_THREADS = 256;
constexpr int TU_MAXK = 128;

template <int NC>
__global__ void __launch_bounds__(TU_THREADS)
ts_update_kernel(const double2 *__restrict__ V, int kv, const double2 *__restrict__ Y, int ldy,
                 int c0, const double2 *IN, double2 *OUT, int beta_one, double sign,
                 long long n, const int *__restrict__ status) {
  if (status != nullptr && *status != 0) return;
  __shared__ double2 Ys[TU_MAXK * NC];
  for (int e = threadIdx.x; e < kv * NC; e += blockDim.x) {
    const int j = e / NC, c = e % NC;
    Ys[e] = cscale(sign, Y[(long long)j * ldy + c0 + c]);
  }
  __syncthreads();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    double2 acc[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) acc[c] = make_double2(0.0, 0.0);
    for (int j = 0; j < kv; ++j) {
      const double2 v = __ldg(V + (long long)j * n + i);
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[c] = cfma(v, Ys[j * NC + c], acc[c]);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const long long o = (long long)(c0 + c) * n + i;
      OUT[o] = beta_one ? cadd(IN[o], acc[c]) : acc[c];
    }
  }
}

cudaError_t launch_ts_update(const double2 *V, int kv, const double2 *Y, int ldy, int ncol,
                             const double2 *IN, double2 *OUT, int beta_one, double sign,
                             long long n, const int *status, cudaStream_t s) {
  ProfLaunch prof_(PC_TS, s);
  if (kv > TU_MAXK || kv < 1 || ncol < 1) return cudaErrorInvalidValue;
  long long blocks = (n + TU_THREADS - 1) / TU_THREADS;
  if (blocks > 1216) blocks = 1216;
  for (int c0 = 0; c0 < ncol;) {
    const int rem = ncol - c0;
    const int nc = rem >= 16 ? 16 : rem >= 8 ? 8 : rem >= 4 ? 4 : rem >= 2 ? 2 : 1;
    dim3 grid((unsigned)blocks);
    switch (nc) {
      case 16: ts_update_kernel<16><<<grid, TU_THREADS, 0, s>>>(V, kv, Y, ldy, c0, IN, OUT, beta_one, sign, n, status); break;
      case 8: ts_update_kernel<8><<<grid, TU_THREADS, 0, s>>>(V, kv, Y, ldy, c0, IN, OUT, beta_one, sign, n, status); break;
      case 4: ts_update_kernel<4><<<grid, TU_THREADS, 0, s>>>(V, kv, Y, ldy, c0, IN, OUT, beta_one, sign, n, status); break;
      case 2: ts_update_kernel<2><<<grid, TU_THREADS, 0, s>>>(V, kv, Y, ldy, c0, IN, OUT, beta_one, sign, n, status); break;
      default: ts_update_kernel<1><<<grid, TU_THREADS, 0, s>>>(V, kv, Y, ldy, c0, IN, OUT, beta_one, sign, n, status); break;
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    c0 += nc;
  }
  return cudaSuccess;
}

// ----------------------------------------------------------------- Arnoldi helpers

__global__ void arnoldi_normalize_finalize_kernel(const double *pw, int nb,
                                                  const double *pw0, int nb0,
                                                  double2 *H, int ldh, int j, double lucky,
                                                  int *status, int *m_eff) {
  chain_enter();
  if (*status != 0) return;
  double a[1] = {0.0}, b[1] = {0.0};
  for (int i = threadIdx.x; i < nb; i += blockDim.x) a[0] += pw[(long long)i * 2];
  for (int i = threadIdx.x; i < nb0; i += blockDim.x) b[0] += pw0[(long long)i * 3 + 2];
  block_sum<1>(a);
  block_sum<1>(b);
  if (threadIdx.x == 0) {
    const double hn = sqrt(a[0]);
    H[(long long)(j + 1) * ldh + j] = make_double2(hn, 0.0);
    if (hn <= lucky * sqrt(b[0])) {
      *status = 1;
      *m_eff = j + 1;
    }
  }
}

cudaError_t launch_arnoldi_normalize_finalize(const double *partial_w, int nb,
                                              const double *partial_w0, int nb0, double2 *H,
                                              int ldh, int j, double lucky, int *status,
                                              int *m_eff, cudaStream_t s) {
  ProfLaunch prof_(PC_STREAM, s);
  return launch_chained(arnoldi_normalize_finalize_kernel, dim3(1), dim3(256), 0, s, partial_w, nb, partial_w0, nb0, H,
                        ldh, j, lucky, status, m_eff);
}

__global__ void norm_finalize_kernel(const double *__restrict__ partial, int nb, int stride,
                                     double2 *dst) {
  double a[1] = {0.0};
  for (int i = threadIdx.x; i < nb; i += blockDim.x) a[0] += partial[(long long)i * stride];
  block_sum<1>(a);
  if (threadIdx.x == 0) *dst = make_double2(sqrt(a[0]), 0.0);
}

cudaError_t launch_norm_finalize(const double *partial, int nb, int stride, double2 *dst,
                                 cudaStream_t s) {
  ProfLaunch prof_(PC_STREAM, s);
  norm_finalize_kernel<<<1, 256, 0, s>>>(partial, nb, stride, dst);
  return cudaGetLastError();
}

}  // namespace wd
