// fp64 GMRES-based iterative refinement (section "Algorithmic Framework":
// x0 from the low-precision factors, then GMRES with the factors as a left
// preconditioner, fp64 working precision, at most 50 iterations, HPL
// backward-error criterion below 16).
//
// Kernels:
//   gemv_partial / gemv_finish  r = b - A x for up to 8 columns; A (fp64,
//       column major) is read once for all columns, coalesced 16-byte loads,
//       split over column chunks with a deterministic second pass.  The
//       first pass can also accumulate |A| row sums (||A||_inf).
//   (the preconditioner z = U^{-1} L^{-1} v is in precond.cu)
//   mgs_step / vec_norm / givens / cycle_start / cycle_finish / update:
//       modified Gram-Schmidt Arnoldi, Givens least squares, x += V y.
// All control decisions are taken on the device; the host reads a few
// words per Arnoldi step to decide whether to launch the next one.
#include "internal.h"

#include <string.h>

#include <algorithm>
#include <mutex>
#include <vector>

namespace hpmxp {
namespace {

constexpr int kMaxM = 64;     // largest restart length
constexpr int kMaxK = 8;      // right-hand sides refined together
constexpr int kRedBlocks = 304;

__device__ inline unsigned long long dbits(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ inline double bits_d(unsigned long long b) { return __longlong_as_double((long long)b); }

// |a| as an fp32 lower bound from the top word of the fp64 pattern (exponent
// rebias, 20 mantissa bits, tiny values flushed to 0): integer ops only, so
// the ||A||_inf estimate of the stopping test costs no fp64 instructions.
__device__ inline float abs_f32_est(double a) {
  const int hi = __double2hiint(a) & 0x7fffffff;
  const int t = hi - (896 << 20);
  return t > 0 ? __int_as_float(min(t, 0x7f7fffff >> 3) << 3) : 0.0f;
}

// fp64 -> fp32 truncated toward zero, integer operations only (exponent
// rebias and the top 23 mantissa bits; values below the fp32 normal range
// flush to zero, which the generated systems never produce).
__device__ inline float trunc_f32(double a) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(a);
  const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
  const int e = (int)((hi >> 20) & 0x7ff) - 896;          // fp32 biased exponent
  const uint32_t mant = ((hi & 0xfffffu) << 3) | (lo >> 29);
  const uint32_t sign = hi & 0x80000000u;
  return e > 0 ? __uint_as_float(sign | ((uint32_t)min(e, 255) << 23) | mant) : __uint_as_float(sign);
}

// ---------------------------------------------------------------------------
// Per right-hand-side state of the refinement (device memory).
// ---------------------------------------------------------------------------
struct RhsState {
  double H[(kMaxM + 1) * kMaxM];   // Hessenberg, column major (m+1) x m
  double cs[kMaxM], sn[kMaxM], g[kMaxM + 1], y[kMaxM];
  double beta, tol, sr, hn;
  double anorm, bnorm;
  unsigned long long rn_bits, xn_bits, bn_bits, an_bits;   // max-reductions (non-negative doubles)
  int outer_active;   // refinement still running
  int cycle_active;   // inside a GMRES cycle, Arnoldi steps still wanted
  int k;              // Arnoldi steps done in the current cycle
  int iters, outer, status;
};

struct Brief {          // copied to the host after each control kernel
  int outer_active, cycle_active, iters, outer, status;
  int pad;
  double sr;
};

// What the host reads in one copy: the status word and the briefs.
struct Report {
  uint32_t status;
  uint32_t pad[15];
  Brief brief[kMaxK];
};

struct SolveParams {
  int n_rhs, m, max_iters;
  double inner_tol, theta, accept;
  int64_t n;
};

// ---------------------------------------------------------------------------
// GEMV: P[c][i + r*n] = sum_{j in chunk c} A(i, j) X(j, r); optional |A| row
// sums (fp32 estimate or exact fp64) into RS[c][i].
// 256 threads x 2 rows = 512 rows per CTA; the chunk's X is staged in shared
// memory once; each thread keeps 8 independent 16-byte column loads in
// flight (HBM bytes in flight per SM is what bounds this kernel).
// ---------------------------------------------------------------------------
constexpr int kGemvRows = 512;
constexpr int kGemvThreads = 256;
constexpr int kGemvChunkElems = 4096;   // columns x right-hand sides staged per CTA

template <int K, int kAbs, bool kF32 = false>   // kAbs: 0 none, 1 fp32 estimate, 2 fp64 exact
__global__ void __launch_bounds__(kGemvThreads) gemv_partial_kernel(int64_t n, const double* __restrict__ A,
                                                                    int64_t lda, const double* __restrict__ X,
                                                                    int64_t ldx, int64_t chunk,
                                                                    float* __restrict__ A32, int64_t ld32,
                                                                    double* __restrict__ P, void* __restrict__ RS,
                                                                    Gate gate) {
  pdl_wait();
  pdl_trigger();
  if (gate.closed()) return;
  __shared__ double xs[kGemvChunkElems];   // xs[r * chunk + jj]
  const int64_t i = (int64_t)blockIdx.x * kGemvRows + 2 * threadIdx.x;
  const int64_t j0 = (int64_t)blockIdx.y * chunk, j1 = min(j0 + chunk, n);
  const int cnt = (int)(j1 - j0);
  for (int t = threadIdx.x; t < cnt * K; t += kGemvThreads) {
    const int jj = t % cnt, r = t / cnt;
    xs[r * chunk + jj] = X[j0 + jj + r * ldx];
  }
  __syncthreads();
  if (i >= n) return;
  double acc0[K], acc1[K];
  float facc0[K], facc1[K];
#pragma unroll
  for (int r = 0; r < K; ++r) { acc0[r] = 0.0; acc1[r] = 0.0; facc0[r] = 0.0f; facc1[r] = 0.0f; }
  float s0 = 0.0f, s1 = 0.0f;
  double d0 = 0.0, d1 = 0.0;
  const bool two = i + 1 < n;
  const bool vec = two && ((((uintptr_t)(A + i)) & 15) == 0) && ((lda & 1) == 0);
  const double* col = A + i + j0 * lda;
  // optional copy of the visited entries, truncated to fp32, for the fp32 operator's later products
  float* col32 = A32 ? A32 + i + j0 * ld32 : nullptr;
  auto body = [&](double a0, double a1, int jj) {
    if (kF32) {
      // fp32 operator: A truncated to fp32, products accumulated in fp32
      const float f0 = trunc_f32(a0), f1 = trunc_f32(a1);
#pragma unroll
      for (int r = 0; r < K; ++r) {
        const float xv = (float)xs[r * chunk + jj];
        facc0[r] = __fmaf_rn(f0, xv, facc0[r]);
        facc1[r] = __fmaf_rn(f1, xv, facc1[r]);
      }
    } else {
#pragma unroll
      for (int r = 0; r < K; ++r) {
        const double xv = xs[r * chunk + jj];
        acc0[r] = __fma_rn(a0, xv, acc0[r]);
        acc1[r] = __fma_rn(a1, xv, acc1[r]);
      }
    }
    if (kAbs == 1) { s0 += abs_f32_est(a0); s1 += abs_f32_est(a1); }
    if (kAbs == 2) { d0 += fabs(a0); d1 += fabs(a1); }
  };
  int jj = 0;
  if (vec) {
    for (; jj + 8 <= cnt; jj += 8) {
      double2 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldcs(reinterpret_cast<const double2*>(col + (int64_t)u * lda));
      col += 8 * lda;
      if (col32) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          *reinterpret_cast<float2*>(col32 + (int64_t)u * ld32) = make_float2(trunc_f32(v[u].x), trunc_f32(v[u].y));
        col32 += 8 * ld32;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) body(v[u].x, v[u].y, jj + u);
    }
  }
  for (; jj < cnt; ++jj) {
    const double a0 = col[0], a1 = two ? col[1] : 0.0;
    col += lda;
    if (col32) {
      col32[0] = trunc_f32(a0);
      if (two) col32[1] = trunc_f32(a1);
      col32 += ld32;
    }
    body(a0, a1, jj);
  }
  double* Pc = P + (int64_t)blockIdx.y * n * K;
#pragma unroll
  for (int r = 0; r < K; ++r) {
    Pc[i + r * n] = kF32 ? (double)facc0[r] : acc0[r];
    if (two) Pc[i + 1 + r * n] = kF32 ? (double)facc1[r] : acc1[r];
  }
  if (kAbs == 1) {
    float* R = (float*)RS + (int64_t)blockIdx.y * n;
    R[i] = s0;
    if (two) R[i + 1] = s1;
  } else if (kAbs == 2) {
    double* R = (double*)RS + (int64_t)blockIdx.y * n;
    R[i] = d0;
    if (two) R[i + 1] = d1;
  }
}

// The fp32 operator's product from the fp32 copy of A: the same chunks, the
// same fp32 accumulation over each chunk's columns in order as the fp64-read
// variant (so the same partial sums), 4 rows per thread, 16-byte loads.
constexpr int kGemv32Rows = 4 * kGemvThreads;
template <int K>
__global__ void __launch_bounds__(kGemvThreads) gemv32_partial_kernel(int64_t n, const float* __restrict__ A32,
                                                                      int64_t ld32, const double* __restrict__ X,
                                                                      int64_t ldx, int64_t chunk,
                                                                      double* __restrict__ P, Gate gate) {
  pdl_wait();
  pdl_trigger();
  if (gate.closed()) return;
  __shared__ double xs[kGemvChunkElems];
  const int64_t i = (int64_t)blockIdx.x * kGemv32Rows + 4 * threadIdx.x;
  const int64_t j0 = (int64_t)blockIdx.y * chunk, j1 = min(j0 + chunk, n);
  const int cnt = (int)(j1 - j0);
  for (int t = threadIdx.x; t < cnt * K; t += kGemvThreads) {
    const int jj = t % cnt, r = t / cnt;
    xs[r * chunk + jj] = X[j0 + jj + r * ldx];
  }
  __syncthreads();
  if (i >= n) return;
  const int rows = (int)min((int64_t)4, n - i);
  float acc[4][K];
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int r = 0; r < K; ++r) acc[q][r] = 0.0f;
  const float* col = A32 + i + j0 * ld32;
  int jj = 0;
  if (rows == 4) {
    for (; jj + 8 <= cnt; jj += 8) {
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldcs(reinterpret_cast<const float4*>(col + (int64_t)u * ld32));
      col += 8 * ld32;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float a[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int r = 0; r < K; ++r) {
          const float xv = (float)xs[r * chunk + jj + u];
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[q][r] = __fmaf_rn(a[q], xv, acc[q][r]);
        }
      }
    }
  }
  for (; jj < cnt; ++jj) {
#pragma unroll
    for (int r = 0; r < K; ++r) {
      const float xv = (float)xs[r * chunk + jj];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < rows) acc[q][r] = __fmaf_rn(col[q], xv, acc[q][r]);
    }
    col += ld32;
  }
  double* Pc = P + (int64_t)blockIdx.y * n * K;
#pragma unroll
  for (int r = 0; r < K; ++r)
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < rows) Pc[i + q + r * n] = (double)acc[q][r];
}

// out(i, r) = B(i, r) - sum_c P[c](i, r), or + sum_c P[c](i, r) when B is NULL
// (chunks in order); max-reduces
// |out|, |X| (when xn) and the row sums (when abs_mode) into the states.
// One right-hand side per grid row; eight threads share a row's chunks (a small
// system's few rows would otherwise wait for each load in turn: 6.0 us at n =
// 1024, 67 us at 8192 with eight right-hand sides) and are summed in order; the
// rows' maxima by shuffles, one atomic per CTA and maximum.
// With `redo`, the status word of a call that cannot report it: a set timeout bit
// says that the partial sums are void, and the rows are summed here from A and X
// by fp64 FMAs instead (the same eight threads, every eighth column each).
__device__ inline unsigned long long warp_max(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
constexpr int kFinRows = 32, kFinGroups = 8;   // rows of a CTA, threads that share a row's pieces
__global__ void __launch_bounds__(kFinRows * kFinGroups)
gemv_finish_kernel(int64_t n, int K, int nchunk, const double* __restrict__ P, const double* __restrict__ B,
                   int64_t ldb, double* __restrict__ out, int64_t ldo, const double* __restrict__ X, int64_t ldx,
                   int abs_mode, const void* __restrict__ RS, RhsState* st, int track_norms, GemvSplit split, Gate gate,
                   const uint32_t* redo, const double* __restrict__ A, int64_t lda) {
  pdl_wait();
  pdl_trigger();
  if (gate.closed()) return;
  __shared__ double sh[2][kFinGroups][kFinRows];
  const int tx = threadIdx.x % kFinRows, ty = threadIdx.x / kFinRows;
  const int64_t i = (int64_t)blockIdx.x * kFinRows + tx;
  const int r = blockIdx.y;
  const bool in = i < n, rows_too = track_norms && abs_mode && r == 0;
  if (split.ctas) nchunk = split.pieces((int)(min(i, n - 1) / kGemvTileRows));   // the tile's own count
  double s = 0.0, a = 0.0;
  if (in && redo && (*redo & kErrTimeout)) {
    for (int64_t j = ty; j < n; j += kFinGroups) s = __fma_rn(A[i + j * lda], X[j + r * ldx], s);
  } else if (in) {
    for (int c = ty; c < nchunk; c += kFinGroups) s += P[((int64_t)c * K + r) * n + i];
    if (rows_too)
      for (int c = ty; c < nchunk; c += kFinGroups)
        a += abs_mode == 1 ? (double)((const float*)RS)[(int64_t)c * n + i] : ((const double*)RS)[(int64_t)c * n + i];
  }
  sh[0][ty][tx] = s;
  sh[1][ty][tx] = a;
  __syncthreads();
  if (ty != 0) return;
#pragma unroll
  for (int g = 1; g < kFinGroups; ++g) {
    s += sh[0][g][tx];
    a += sh[1][g][tx];
  }
  const double v = B && in ? B[i + r * ldb] - s : s;
  if (in) out[i + r * ldo] = v;
  if (!track_norms) return;
  const unsigned long long rn = warp_max(in ? dbits(fabs(v)) : 0ull);
  const unsigned long long xn = warp_max(in ? dbits(fabs(X[i + r * ldx])) : 0ull);
  const unsigned long long bn = B ? warp_max(in ? dbits(fabs(B[i + r * ldb])) : 0ull) : 0ull;
  const unsigned long long an = rows_too ? warp_max(dbits(a)) : 0ull;
  if (tx == 0) {
    atomicMax(&st[r].rn_bits, rn);
    atomicMax(&st[r].xn_bits, xn);
    if (B) atomicMax(&st[r].bn_bits, bn);
    if (rows_too)
      for (int k = 0; k < K; ++k) atomicMax(&st[k].an_bits, an);
  }
}

// ---------------------------------------------------------------------------
// Vector kernels.  Deterministic reductions: per-thread strided partials,
// fixed-shape block tree, per-block partials summed the same way by the last CTA.
// ---------------------------------------------------------------------------
// The sum of v over the block (a multiple of 32 threads), the same for every
// thread: warps by shuffles, then their sums by each warp.
__device__ inline double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ inline double block_sum(double v, double* sh) {
  const int lane = threadIdx.x & 31;
  v = warp_sum(v);
  if (lane == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  v = warp_sum(lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0);
  __syncthreads();
  return v;
}

// For every rhs r that is in an active cycle: optionally w -= h_prev v_prev
// (h_prev = H(i-1, j)), then reduce either <w, v_i> (into H(i, j)) or <w, w>
// (into hn, as a square root) when i == j + 1.
__global__ void __launch_bounds__(256) mgs_kernel(int64_t n, int K, int m, int j, int i, double* W, int64_t ldw,
                                                  const double* V, int64_t ldv_col, int64_t ldv_rhs,
                                                  RhsState* st, double* partials, unsigned int* counter, Gate gate) {
  pdl_wait();
  pdl_trigger();
  if (gate.closed()) return;
  __shared__ double sh[32];
  __shared__ bool last;
  for (int r = 0; r < K; ++r) {
    const bool act = st[r].cycle_active != 0;
    double part = 0.0;
    if (act) {
      double* w = W + r * ldw;
      const double* vprev = i > 0 ? V + r * ldv_rhs + (int64_t)(i - 1) * ldv_col : nullptr;
      const double hprev = i > 0 ? st[r].H[(i - 1) + j * (m + 1)] : 0.0;
      const double* vi = i <= j ? V + r * ldv_rhs + (int64_t)i * ldv_col : nullptr;
      for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        double wt = w[t];
        if (vprev) { wt = __fma_rn(-hprev, vprev[t], wt); w[t] = wt; }
        part = vi ? __fma_rn(wt, vi[t], part) : __fma_rn(wt, wt, part);
      }
    }
    const double bs = block_sum(part, sh);
    if (threadIdx.x == 0) partials[(int64_t)r * kRedBlocks + blockIdx.x] = bs;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int r = 0; r < K; ++r) {
    if (!st[r].cycle_active) continue;
    double s = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) s += partials[(int64_t)r * kRedBlocks + b];
    s = block_sum(s, sh);
    if (threadIdx.x == 0) {
      if (i <= j) st[r].H[i + j * (m + 1)] = s;
      else st[r].hn = sqrt(s);
    }
  }
  if (threadIdx.x == 0) *counter = 0;
}

// The tail of Arnoldi step j, one CTA per right-hand side, for systems small
// enough that one SM streams w and the basis faster than j + 4 launches would
// start: modified Gram-Schmidt (for i = 0 .. j, H(i, j) = <w, v_i> then w -=
// H(i, j) v_i, and hn = ||w||), the Givens update, and v_{j+1} = w / hn.  Every
// entry of w sees the same operations as in mgs_kernel; the dot products are
// summed by this CTA's fixed tree instead of across CTAs.
__device__ void givens_rhs(const SolveParams& sp, int j, RhsState* st, Brief* brief, int r);
constexpr int kFusedMgsThreads = 1024;
constexpr int64_t kFusedMgsMaxElems = 16384;   // n * K at most
__global__ void __launch_bounds__(kFusedMgsThreads) arnoldi_tail_kernel(SolveParams sp, int64_t n, int m, int j,
                                                                        double* W, int64_t ldw, double* V,
                                                                        int64_t ldv_col, int64_t ldv_rhs,
                                                                        RhsState* st, Brief* brief) {
  pdl_wait();
  pdl_trigger();
  __shared__ double sh[32];
  const int r = blockIdx.x;
  if (st[r].cycle_active) {   // the same value for every thread
    double* w = W + r * ldw;
    double hprev = 0.0;
    for (int i = 0; i <= j + 1; ++i) {
      const double* vprev = i > 0 ? V + r * ldv_rhs + (int64_t)(i - 1) * ldv_col : nullptr;
      const double* vi = i <= j ? V + r * ldv_rhs + (int64_t)i * ldv_col : nullptr;
      double part = 0.0;
      for (int64_t t = threadIdx.x; t < n; t += kFusedMgsThreads) {
        double wt = w[t];
        if (vprev) { wt = __fma_rn(-hprev, vprev[t], wt); w[t] = wt; }
        part = vi ? __fma_rn(wt, vi[t], part) : __fma_rn(wt, wt, part);
      }
      const double s = block_sum(part, sh);
      if (threadIdx.x == 0) {
        if (i <= j) st[r].H[i + j * (m + 1)] = s;
        else st[r].hn = sqrt(s);
      }
      hprev = s;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) givens_rhs(sp, j, st, brief, r);
  __syncthreads();
  if (!st[r].cycle_active) return;
  const double hn = st[r].hn;
  const double* w = W + r * ldw;
  double* v = V + r * ldv_rhs + (int64_t)(j + 1) * ldv_col;
  for (int64_t t = threadIdx.x; t < n; t += kFusedMgsThreads) v[t] = w[t] / hn;
}

// ||z||_2 for cycle start (beta), into st[r].beta, for rhs with outer_active.
__global__ void __launch_bounds__(256) norm2_kernel(int64_t n, int K, const double* Z, int64_t ldz, RhsState* st,
                                                    double* partials, unsigned int* counter) {
  pdl_wait();
  pdl_trigger();
  __shared__ double sh[32];
  __shared__ bool last;
  for (int r = 0; r < K; ++r) {
    double part = 0.0;
    if (st[r].outer_active) {
      const double* z = Z + r * ldz;
      for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        part = __fma_rn(z[t], z[t], part);
    }
    const double bs = block_sum(part, sh);
    if (threadIdx.x == 0) partials[(int64_t)r * kRedBlocks + blockIdx.x] = bs;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int r = 0; r < K; ++r) {
    double s = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) s += partials[(int64_t)r * kRedBlocks + b];
    s = block_sum(s, sh);
    if (threadIdx.x == 0) st[r].beta = sqrt(s);
  }
  if (threadIdx.x == 0) *counter = 0;
}

// dst(:, r) = src(:, r) / d_r with d_r = st[r].beta (which == 0) or st[r].hn (which == 1),
// for rhs whose flag (cycle_active or outer_active) is set.
__global__ void scale_kernel(int64_t n, int K, const double* src, int64_t lds, double* dst, int64_t ldd,
                             const RhsState* st, int which) {
  pdl_wait();
  pdl_trigger();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  for (int r = 0; r < K; ++r) {
    const bool act = which == 0 ? st[r].outer_active != 0 : st[r].cycle_active != 0;
    if (!act) continue;
    const double d = which == 0 ? st[r].beta : st[r].hn;
    dst[t + r * ldd] = src[t + r * lds] / d;
  }
}

__global__ void init_kernel(int K, RhsState* st) {
  if ((int)threadIdx.x < K) st[threadIdx.x].outer_active = 1;
}

// Outer check: scaled residual from the max-reductions; decide per rhs.
__global__ void check_kernel(SolveParams sp, RhsState* st, Brief* brief, int first) {
  pdl_wait();
  pdl_trigger();
  const int r = threadIdx.x;
  if (r >= sp.n_rhs) return;
  RhsState& s = st[r];
  if (first) {
    s.anorm = bits_d(s.an_bits);
    s.bnorm = bits_d(s.bn_bits);
  }
  if (s.outer_active) {
    const double rn = bits_d(s.rn_bits), xn = bits_d(s.xn_bits);
    const double sr = rn / ((s.anorm * xn + s.bnorm) * ((double)sp.n * 0x1p-53));
    s.sr = sr;
    if (!isfinite(sr)) { s.status = HPMXP_EBREAKDOWN; s.outer_active = 0; }
    else if (sr < sp.accept) { s.status = HPMXP_OK; s.outer_active = 0; }
    else if (s.iters >= sp.max_iters) { s.status = HPMXP_ENOCONV; s.outer_active = 0; }
  }
  s.rn_bits = 0; s.xn_bits = 0;
  s.cycle_active = 0;
  brief[r].outer_active = s.outer_active; brief[r].cycle_active = 0;
  brief[r].iters = s.iters; brief[r].outer = s.outer; brief[r].status = s.status; brief[r].sr = s.sr;
}

// Cycle start (after beta = ||M^{-1} r||): g = beta e1, tolerance.
__global__ void cycle_start_kernel(SolveParams sp, RhsState* st, Brief* brief) {
  pdl_wait();
  pdl_trigger();
  const int r = threadIdx.x;
  if (r >= sp.n_rhs) return;
  RhsState& s = st[r];
  s.cycle_active = 0;
  if (s.outer_active) {
    if (!(isfinite(s.beta) && s.beta > 0.0)) {
      s.status = HPMXP_EBREAKDOWN; s.outer_active = 0;
    } else {
      s.outer += 1;
      s.k = 0;
      for (int t = 0; t <= sp.m; ++t) s.g[t] = 0.0;
      s.g[0] = s.beta;
      const double adapt = sp.theta > 0.0 ? sp.theta * sp.accept / s.sr : 0.0;
      s.tol = s.beta * fmax(sp.inner_tol, adapt);
      s.cycle_active = s.iters < sp.max_iters ? 1 : 0;
    }
  }
  brief[r].outer_active = s.outer_active; brief[r].cycle_active = s.cycle_active;
  brief[r].status = s.status; brief[r].iters = s.iters; brief[r].outer = s.outer; brief[r].sr = s.sr;
}

// Givens update of column j (after MGS filled H(0..j, j) and hn).
// Givens update of right-hand side r after Arnoldi step j (thread r)
__device__ void givens_rhs(const SolveParams& sp, int j, RhsState* st, Brief* brief, int r) {
  RhsState& s = st[r];
  if (s.cycle_active) {
    const int ld = sp.m + 1;
    double* h = s.H + j * ld;
    const double hn = s.hn;
    h[j + 1] = hn;
    for (int i = 0; i < j; ++i) {
      const double a0 = h[i], a1 = h[i + 1];
      h[i] = s.cs[i] * a0 + s.sn[i] * a1;
      h[i + 1] = -s.sn[i] * a0 + s.cs[i] * a1;
    }
    const double hj = h[j];
    const double den = hypot(hj, hn);
    if (!(isfinite(den) && den != 0.0)) {
      s.status = HPMXP_EBREAKDOWN; s.outer_active = 0; s.cycle_active = 0;
    } else {
      s.cs[j] = hj / den;
      s.sn[j] = hn / den;
      h[j] = den;
      h[j + 1] = 0.0;
      s.g[j + 1] = -s.sn[j] * s.g[j];
      s.g[j] = s.cs[j] * s.g[j];
      s.iters += 1;
      s.k = j + 1;
      if (hn == 0.0 || fabs(s.g[j + 1]) <= s.tol || s.k >= sp.m || s.iters >= sp.max_iters) s.cycle_active = 0;
      if (!isfinite(s.g[j + 1])) { s.status = HPMXP_EBREAKDOWN; s.outer_active = 0; s.cycle_active = 0; }
    }
  }
  brief[r].cycle_active = s.cycle_active; brief[r].outer_active = s.outer_active;
  brief[r].iters = s.iters; brief[r].status = s.status;
}
__global__ void givens_kernel(SolveParams sp, int j, RhsState* st, Brief* brief) {
  pdl_wait();
  pdl_trigger();
  if ((int)threadIdx.x < sp.n_rhs) givens_rhs(sp, j, st, brief, threadIdx.x);
}

// y = H(0:k, 0:k)^{-1} g(0:k) by back substitution.
__global__ void cycle_finish_kernel(SolveParams sp, RhsState* st) {
  pdl_wait();
  pdl_trigger();
  const int r = threadIdx.x;
  if (r >= sp.n_rhs) return;
  RhsState& s = st[r];
  if (!s.outer_active) { s.k = 0; return; }
  const int ld = sp.m + 1;
  for (int i = s.k - 1; i >= 0; --i) {
    double acc = s.g[i];
    for (int t = i + 1; t < s.k; ++t) acc = __fma_rn(-s.H[i + t * ld], s.y[t], acc);
    s.y[i] = acc / s.H[i + i * ld];
  }
}

// x(:, r) += V_r(:, 0:k) y_r
__global__ void update_kernel(int64_t n, int K, double* X, int64_t ldx, const double* V, int64_t ldv_col,
                              int64_t ldv_rhs, const RhsState* st) {
  pdl_wait();
  pdl_trigger();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n) return;
  for (int r = 0; r < K; ++r) {
    const int k = st[r].outer_active ? st[r].k : 0;
    double xv = X[t + r * ldx];
    for (int i = 0; i < k; ++i) xv = __fma_rn(V[r * ldv_rhs + (int64_t)i * ldv_col + t], st[r].y[i], xv);
    X[t + r * ldx] = xv;
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
struct SolveWs {
  Report* report;    // the solve's words for the host; status and brief point into it
  uint32_t* status;
  RhsState* st;
  Brief* brief;
  unsigned int* counter;
  size_t control_bytes;   // report .. counter, zeroed at the start of a solve
  bool pdl;               // programmatic launches (launch_vec): not where the call shares the chip
  double* partials;  // kMaxK * kRedBlocks
  double* r;         // n x K
  double* w;         // n x K
  double* tmp;       // n x K
  double* V;         // K x (m+1) x n
  double* P;         // nchunk x n x K
  void* RS;          // nchunk x n (fp64 size)
  void* pub;         // 2 sweeps x round_up(n, 128) x K values x (1 or 2) 8-byte tagged words
  void* dinv;        // inverted diagonal blocks of L and U (precond.cu)
  void* chain;       // the blocks next to them, multiplied by the inverses
  float* a32;        // optional fp32 copy of A (ld32), written by the first residual, NULL if none
  int64_t ld32;
  size_t bytes;
};

// Column chunks of the GEMV: each chunk's X (chunk x K doubles) fits the
// CTA's staging buffer; there are enough CTAs to keep every SM loaded (about
// 8 per SM), but no CTA reads fewer than 32 columns (128 KB of A), so a small
// system does not spread a short product over every SM.
int gemv_chunks(int64_t n, int K = kMaxK) {
  const int64_t rb = cdiv<int64_t>(n, kGemvRows);
  const int64_t spread = std::min<int64_t>(cdiv<int64_t>(8 * 152, rb), cdiv<int64_t>(n, 32));
  int64_t c = std::max<int64_t>(cdiv<int64_t>(n, kGemvChunkElems / K), spread);   // chunk = ceil(n / c) columns
  c = std::max<int64_t>(1, std::min<int64_t>(c, cdiv<int64_t>(n, 8)));
  return (int)c;
}

SolveWs carve_solve(void* base, int64_t n, int64_t K, int m) {
  SolveWs w{};
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = base ? (char*)base + off : nullptr;
    off += round_up<size_t>(bytes, 256);
    return p;
  };
  const int nchunk = gemv_chunks(n);
  w.report = (Report*)take(sizeof(Report));
  w.status = (uint32_t*)w.report;
  w.brief = base ? w.report->brief : nullptr;
  w.st = (RhsState*)take(sizeof(RhsState) * kMaxK);
  w.counter = (unsigned int*)take(256);
  w.control_bytes = off;
  w.partials = (double*)take(sizeof(double) * kMaxK * kRedBlocks);
  w.r = (double*)take(sizeof(double) * n * K);
  w.w = (double*)take(sizeof(double) * n * K);
  w.tmp = (double*)take(sizeof(double) * n * K);
  w.V = (double*)take(sizeof(double) * n * (m + 1) * K);
  w.P = (double*)take(sizeof(double) * nchunk * n * K);
  w.RS = take(sizeof(double) * nchunk * n);
  w.pub = take(precond_pub_bytes(n, K));
  w.dinv = take(precond_inverse_bytes(n));
  w.chain = take(precond_chain_bytes(n));
  w.pdl = sm_budget() <= 0;   // under a budget the call shares the chip, as a batch's systems do
  w.bytes = off;
  return w;
}

// abs_mode: 0 plain, 1 with the fp32 |A| estimate (the first residual; also
// fills w.a32 when there is one), 2 exact |A| row sums, 3 the fp32 operator's
// product (from w.a32 when there is one)
template <int K>
cudaError_t gemv_k(int64_t n, const double* A, int64_t lda, const double* X, int64_t ldx, int abs_mode,
                   const SolveWs& w, int nchunk, cudaStream_t st, Gate gate) {
  const int64_t chunk = cdiv<int64_t>(n, nchunk);
  if (chunk * K > kGemvChunkElems) return cudaErrorInvalidValue;   // gemv_chunks never gives that
  dim3 grid((unsigned)cdiv<int64_t>(n, kGemvRows), (unsigned)nchunk);
  const int T = kGemvThreads;
  double* P = w.P;
  void* RS = w.RS;
  if (abs_mode == 3 && w.a32) {
    dim3 g32((unsigned)cdiv<int64_t>(n, kGemv32Rows), (unsigned)nchunk);
    launch_vec(w.pdl, gemv32_partial_kernel<K>, g32, dim3(T), 0, st, n, w.a32, w.ld32, X, ldx, chunk, P, gate);
  } else if (abs_mode == 3) {
    launch_vec(w.pdl, gemv_partial_kernel<K, 0, true>, grid, dim3(T), 0, st, n, A, lda, X, ldx, chunk, nullptr, 0, P, RS,
               gate);
  } else if (abs_mode == 0) {
    launch_vec(w.pdl, gemv_partial_kernel<K, 0>, grid, dim3(T), 0, st, n, A, lda, X, ldx, chunk, nullptr, 0, P, RS, gate);
  } else if (abs_mode == 1) {
    launch_vec(w.pdl, gemv_partial_kernel<K, 1>, grid, dim3(T), 0, st, n, A, lda, X, ldx, chunk, w.a32, w.ld32, P, RS, gate);
  } else {
    launch_vec(w.pdl, gemv_partial_kernel<K, 2>, grid, dim3(T), 0, st, n, A, lda, X, ldx, chunk, nullptr, 0, P, RS, gate);
  }
  return cudaGetLastError();
}

// The digits share the row-sum scratch (fp64, gemv_chunks(n) per row) with the fp32
// row sums of the product's own pieces, which come first.
size_t gemv_tc_row_sums(int64_t n, const GemvSplit& s) { return round_up<size_t>(sizeof(float) * (size_t)most_of(s) * n, 256); }

// Which products go to the tensor cores (gemv_tc.cu): fp64 ones that do not
// also copy A to fp32, from the order at which two launches for X's digits and
// up to 223 KB of shared memory per SM pay.  Whole residuals timed, microseconds,
// digit products / fp64 FMAs: one right-hand side 47 / 50 at n = 4096, 61 / 70 at
// 5120, 112 / 127 at 8192, 1460 / 1787 at 32768; two 27.5 / 26.4 at 2048, 38 / 45 at
// 3072, 116 / 236 at 8192; four 32 / 43 at 2048; six 32 / 34 at 1024; eight 36 / 43 at
// 1024, 150 / 890 at 8192, 1820 / 13800 at 32768.
bool gemv_on_tensor_cores(int64_t n, int K, const double* A, int64_t lda, int abs_mode, const SolveWs& w,
                          GemvSplit* split) {
  const int64_t min_n = K == 1 ? 4096 : K < 6 ? 2048 : 1024;
  if (!(abs_mode == 0 || (abs_mode == 1 && !w.a32)) || n < min_n) return false;
  const size_t cap = (size_t)gemv_chunks(n);
  GemvSplit s;
  if (!gemv_tc_split(n, A, lda, (int)cap, &s)) return false;
  if (gemv_tc_row_sums(n, s) + gemv_tc_bytes(n) > sizeof(double) * cap * n) return false;
  *split = s;
  return true;
}

// out = b - A X (b may be NULL: out = A X), with optional norm tracking.  live:
// the right-hand sides whose columns are wanted (none given: all; out's others are
// unspecified).  redo: for a caller that does not read w.status, make a void
// product good (without norms).
cudaError_t residual(int64_t n, int K, const double* A, int64_t lda, const double* X, int64_t ldx,
                     const double* B, int64_t ldb, double* out, int64_t ldo, int abs_mode, int track,
                     const SolveWs& w, cudaStream_t st, Gate gate = {}, Gate live = {},
                     bool redo = false) {
  int nchunk = gemv_chunks(n, K);
  cudaError_t e;
  void* tok = prof_begin(st);
  GemvSplit split;
  if (gemv_on_tensor_cores(n, K, A, lda, abs_mode, w, &split)) {
    void* prep = (char*)w.RS + gemv_tc_row_sums(n, split);
    e = gemv_tc(n, K, A, lda, X, ldx, abs_mode == 1, prep, w.P, w.RS, split, w.status, st, w.pdl, gate,
                live);
  } else {
    switch (K) {
      case 1: e = gemv_k<1>(n, A, lda, X, ldx, abs_mode, w, nchunk, st, gate); break;
      case 2: e = gemv_k<2>(n, A, lda, X, ldx, abs_mode, w, nchunk, st, gate); break;
      case 3: e = gemv_k<3>(n, A, lda, X, ldx, abs_mode, w, nchunk, st, gate); break;
      case 4: e = gemv_k<4>(n, A, lda, X, ldx, abs_mode, w, nchunk, st, gate); break;
      case 5: e = gemv_k<5>(n, A, lda, X, ldx, abs_mode, w, nchunk, st, gate); break;
      case 6: e = gemv_k<6>(n, A, lda, X, ldx, abs_mode, w, nchunk, st, gate); break;
      case 7: e = gemv_k<7>(n, A, lda, X, ldx, abs_mode, w, nchunk, st, gate); break;
      default: e = gemv_k<8>(n, A, lda, X, ldx, abs_mode, w, nchunk, st, gate); break;
    }
  }
  if (e != cudaSuccess) return e;
  launch_vec(w.pdl, gemv_finish_kernel, dim3((unsigned)cdiv<int64_t>(n, kFinRows), K), dim3(kFinRows * kFinGroups), 0, st,
             n, K, nchunk, w.P, B, ldb, out, ldo, X, ldx, abs_mode == 3 ? 0 : abs_mode, w.RS, w.st, track, split, gate,
             redo ? (const uint32_t*)w.status : nullptr, A, lda);
  prof_end(tok, abs_mode == 3 ? kProfGemv32 : kProfGemv, 8.0 * (double)n * (double)n, st);
  count_launches(2);
  return cudaGetLastError();
}

struct Solver {
  int64_t n;
  int K, m;
  const double* A; int64_t lda;
  const uint16_t* LU; int64_t ldlu; int fmt;
  const double* rs = nullptr;   // balancing of the factors (NULL: none)
  const double* cs = nullptr;
  const double* B; int64_t ldb;
  double* X; int64_t ldx;
  hpmxp_ir_params prm;
  SolveWs w;
  cudaStream_t st;
  int epoch = 0;
  PrecondPlan plan;
  Report rep;

  size_t report_bytes() const { return offsetof(Report, brief) + sizeof(Brief) * K; }
  // The right-hand sides that still want refinement / Arnoldi steps; as gates of
  // launches issued ahead of the host's knowledge: some still does
  Gate outer_gate() const { return {&w.st->outer_active, K, (int)(sizeof(RhsState) / sizeof(int))}; }
  Gate cycle_gate() const { return {&w.st->cycle_active, K, (int)(sizeof(RhsState) / sizeof(int))}; }

  int64_t ldv_rhs() const { return n * (m + 1); }

  cudaError_t precond(const double* v, int64_t ldv, double* z, int64_t ldz, Gate gate = {}) {
    ++epoch;
    void* tok = prof_begin(st);
    const cudaError_t e = precond_launch(plan, prm.precond_fp32 != 0, K, n, LU, ldlu, fmt, w.dinv, w.chain, v, ldv, z,
                                         ldz, w.pub, epoch, w.status, rs, cs, st, gate);
    prof_end(tok, kProfPrecond, 2.0 * (double)n * (double)n, st);
    count_launches(1);
    return e;
  }

  // CTAs of the reductions over n: no more than hold an entry per thread
  int red_blocks() const { return (int)std::min<int64_t>(kRedBlocks, cdiv<int64_t>(n, 256)); }
  // Arnoldi step j after w = M^{-1} A v_j: modified Gram-Schmidt, the Givens
  // update (into the brief) and v_{j+1}; one launch for small systems, else one
  // launch per projection, then the rotation and the scaling
  void arnoldi_tail(int j, Gate gate) {
    const SolveParams sp{K, m, prm.max_iters, prm.inner_tol, prm.theta, prm.accept, n};
    if (n * K <= kFusedMgsMaxElems) {
      launch_vec(w.pdl, arnoldi_tail_kernel, dim3(K), dim3(kFusedMgsThreads), 0, st, sp, n, m, j, w.w, n, w.V, n,
                 ldv_rhs(), w.st, w.brief);
      count_launches(1);
      return;
    }
    for (int i = 0; i <= j + 1; ++i)
      launch_vec(w.pdl, mgs_kernel, dim3(red_blocks()), dim3(256), 0, st, n, K, m, j, i, w.w, n, w.V, n, ldv_rhs(), w.st,
                 w.partials, w.counter, gate);
    launch_vec(w.pdl, givens_kernel, dim3(1), dim3(32), 0, st, sp, j, w.st, w.brief);
    launch_vec(w.pdl, scale_kernel, dim3((unsigned)cdiv<int64_t>(n, 256)), dim3(256), 0, st, n, K, w.w, n,
               w.V + (int64_t)(j + 1) * n, ldv_rhs(), w.st, 1);
    count_launches(j + 4);
  }
  bool any(int Brief::*f) const {
    for (int r = 0; r < K; ++r)
      if (rep.brief[r].*f) return true;
    return false;
  }

  cudaError_t setup() {
    cudaError_t e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const bool fp32 = prm.precond_fp32 != 0;
    if (!precond_plan(n, K, fp32, sms, sm_budget(), &plan)) return cudaErrorInvalidValue;
    if ((e = cudaMemsetAsync(w.pub, 0, precond_pub_bytes(n, K), st)) != cudaSuccess) return e;
    if ((e = precond_setup(n, LU, ldlu, fmt, fp32, w.dinv, w.chain, st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(w.report, 0, w.control_bytes, st)) != cudaSuccess) return e;
    init_kernel<<<1, 32, 0, st>>>(K, w.st);
    count_launches(1);
    return cudaGetLastError();
  }

  // z = M^{-1} r, beta, v0 = z / beta
  // ahead (here and below): issued before the host knows that it is wanted
  cudaError_t cycle_start(bool ahead) {
    const SolveParams sp{K, m, prm.max_iters, prm.inner_tol, prm.theta, prm.accept, n};
    const cudaError_t e = precond(w.r, n, w.tmp, n, ahead ? outer_gate() : Gate{});
    if (e != cudaSuccess) return e;
    launch_vec(w.pdl, norm2_kernel, dim3(red_blocks()), dim3(256), 0, st, n, K, w.tmp, n, w.st, w.partials, w.counter);
    launch_vec(w.pdl, cycle_start_kernel, dim3(1), dim3(32), 0, st, sp, w.st, w.brief);
    launch_vec(w.pdl, scale_kernel, dim3((unsigned)cdiv<int64_t>(n, 256)), dim3(256), 0, st, n, K, w.tmp, n, w.V,
               ldv_rhs(), w.st, 0);
    count_launches(3);
    return cudaGetLastError();
  }
  // w = M^{-1} (A v_j), orthogonalised; the product in fp32 or fp64 as matvec_fp32 says
  cudaError_t arnoldi_step(int j, bool ahead) {
    const Gate gate = ahead ? cycle_gate() : Gate{};
    cudaError_t e = residual(n, K, A, lda, w.V + (int64_t)j * n, ldv_rhs(), nullptr, 0, w.tmp, n,
                             prm.matvec_fp32 ? 3 : 0, 0, w, st, gate, cycle_gate());
    if (e != cudaSuccess) return e;
    if ((e = precond(w.tmp, n, w.w, n, gate)) != cudaSuccess) return e;
    arnoldi_tail(j, gate);
    return cudaGetLastError();
  }
  // x += V y
  cudaError_t cycle_finish() {
    const SolveParams sp{K, m, prm.max_iters, prm.inner_tol, prm.theta, prm.accept, n};
    launch_vec(w.pdl, cycle_finish_kernel, dim3(1), dim3(32), 0, st, sp, w.st);
    launch_vec(w.pdl, update_kernel, dim3((unsigned)cdiv<int64_t>(n, 256)), dim3(256), 0, st, n, K, X, ldx, w.V, n,
               ldv_rhs(), w.st);
    count_launches(2);
    return cudaGetLastError();
  }
  // r = b - A x, norms; decide
  cudaError_t outer_check(bool first) {
    const SolveParams sp{K, m, prm.max_iters, prm.inner_tol, prm.theta, prm.accept, n};
    const cudaError_t e = residual(n, K, A, lda, X, ldx, B, ldb, w.r, n, first ? 1 : 0, 1, w, st, {}, outer_gate());
    if (e != cudaSuccess) return e;
    launch_vec(w.pdl, check_kernel, dim3(1), dim3(32), 0, st, sp, w.st, w.brief, first ? 1 : 0);
    count_launches(1);
    return cudaGetLastError();
  }

  // The decisions are made on the device (RhsState); the host learns them by
  // reading the report, 15 to 20 us in which the GPU idles.  The first cycle
  // does not wait for the first check, and no cycle's first Arnoldi step waits
  // for the cycle's start: either is wanted as a rule, and its gates close where
  // it is not.  Issuing the later steps ahead as well gained nothing: the step
  // after a cycle's last one costs 25 us (n = 1024) to 90 us with its gates
  // closed.  628 -> 574 us at n = 1024; 24 mixed systems in one batch 9.30 -> 8.83
  // ms.  Where x0 is accepted the closed cycle costs what the wait would have and
  // more: 145 -> 168 us at n = 1024, 802 -> 828 at 4096 in fp64, 803 -> 854 at 8192
  // with eight right-hand sides.  With the kernel timers on, nothing is issued ahead.
  cudaError_t run() {
    const bool ahead = !prof_on();
    auto report = [&] { return read_to_host(&rep, w.report, report_bytes(), st); };
    cudaError_t e = setup();
    if (e != cudaSuccess) return e;
    if ((e = precond(B, ldb, X, ldx)) != cudaSuccess) return e;   // x0 = U^{-1} L^{-1} b
    for (bool first = true;; first = false) {
      if ((e = outer_check(first)) != cudaSuccess) return e;
      if (!(first && ahead)) {   // a later check is the last one as a rule
        if ((e = report()) != cudaSuccess) return e;
        if (!any(&Brief::outer_active)) return cudaSuccess;
      }
      if ((e = cycle_start(first && ahead)) != cudaSuccess) return e;
      if (!ahead) {
        if ((e = report()) != cudaSuccess) return e;
        if (!any(&Brief::outer_active)) return cudaSuccess;
      }
      for (int j = 0; j < m && ((j == 0 && ahead) || any(&Brief::cycle_active)); ++j) {
        if ((e = arnoldi_step(j, j == 0 && ahead)) != cudaSuccess) return e;
        if ((e = report()) != cudaSuccess) return e;
        if (j == 0 && ahead && !any(&Brief::outer_active)) return cudaSuccess;
      }
      if ((e = cycle_finish()) != cudaSuccess) return e;
    }
  }
};

}  // namespace

// Test support: every SM's shared memory filled with `pattern`, so that a
// kernel launched next finds nonzero leftovers there instead of the zeros a
// quiet GPU tends to leave.
__global__ void fill_smem_kernel(uint32_t pattern, uint32_t words) {
  extern __shared__ uint32_t sw[];
  for (uint32_t t = threadIdx.x; t < words; t += blockDim.x) sw[t] = pattern;
  __syncthreads();
  if (sw[(threadIdx.x * 7u) % words] != pattern) asm volatile("" ::: "memory");
}

// Test support: the fp64 decoding of 16-bit factor entries, one per thread.
__global__ void decode16_kernel(const uint16_t* __restrict__ codes, double* __restrict__ out, int64_t count,
                                int fmt) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) out[i] = u16_to_f64(codes[i], fmt);
}

cudaError_t decode16(const uint16_t* codes, double* out, int64_t count, int fmt, cudaStream_t st) {
  if (count <= 0) return cudaSuccess;
  decode16_kernel<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(codes, out, count, fmt);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t fill_smem(uint32_t pattern, cudaStream_t st) {
  int dev = 0, sms = 0, maxb = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&maxb, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fill_smem_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, maxb);
  if (e != cudaSuccess) return e;
  fill_smem_kernel<<<2 * sms, 1024, (size_t)maxb, st>>>(pattern, (uint32_t)maxb / 4);
  count_launches(1);
  return cudaGetLastError();
}

size_t solve_ws_bytes(int64_t n, int64_t nrhs, int restart) { return carve_solve(nullptr, n, nrhs, restart).bytes; }
int64_t a32_ld(int64_t n) { return round_up<int64_t>(n, 4); }
size_t solve_a32_bytes(int64_t n) { return round_up<size_t>(sizeof(float) * (size_t)a32_ld(n) * (size_t)n, 256); }
size_t residual_ws_bytes(int64_t n, int64_t nrhs) { return carve_solve(nullptr, n, nrhs, 1).bytes; }

hpmxp_status solve_ir(int64_t n, const double* A, int64_t lda, const void* LU, int64_t ldlu, int prec,
                      const double* b, int64_t ldb, double* x, int64_t ldx, int64_t nrhs,
                      const hpmxp_ir_params& prm, hpmxp_ir_info* info, void* ws, size_t ws_bytes,
                      cudaStream_t st, const double* rs, const double* cs) {
  Solver s;
  s.n = n; s.K = (int)nrhs; s.m = prm.restart;
  s.A = A; s.lda = lda;
  s.LU = (const uint16_t*)LU; s.ldlu = ldlu; s.fmt = fmt_of(prec);
  s.rs = rs; s.cs = cs;
  s.B = b; s.ldb = ldb; s.X = x; s.ldx = ldx;
  s.prm = prm;
  s.w = carve_solve(ws, n, nrhs, prm.restart);
  // room for the fp32 copy of A after the workspace proper: the fp32 Arnoldi
  // products then read 4 instead of 8 bytes per entry
  if (prm.matvec_fp32 && ws_bytes >= s.w.bytes + solve_a32_bytes(n)) {
    s.w.a32 = (float*)((char*)ws + s.w.bytes);
    s.w.ld32 = a32_ld(n);
  }
  s.st = st;
  cudaError_t e = s.run();
  if (e != cudaSuccess) return status_from_cuda(e);
  if (s.rep.status) return status_from_word(s.rep.status);
  int worst = HPMXP_OK;
  for (int r = 0; r < s.K; ++r) {
    if (info) {
      info[r].iters = s.rep.brief[r].iters;
      info[r].outer = s.rep.brief[r].outer;
      info[r].scaled_resid = s.rep.brief[r].sr;
      info[r].status = s.rep.brief[r].status;
      info[r].reserved = 0;
    }
    if (s.rep.brief[r].status != HPMXP_OK && worst == HPMXP_OK) worst = s.rep.brief[r].status;
  }
  return (hpmxp_status)worst;
}

// ---------------------------------------------------------------------------
// Batched GMRES-IR: every system's refinement as a state machine (the phases
// of Solver::run), advanced in lockstep.  Each round issues every active
// system's next phase on its stream (systems spread over a pool of streams,
// so small systems' kernels run side by side) with an asynchronous copy of its
// brief, then waits once per system and decides every next phase on the host:
// one host decision point per phase for the whole batch.
// ---------------------------------------------------------------------------
namespace {
constexpr int kPoolStreams = 8;

struct StreamPool {
  std::mutex mu;
  bool ok = false;
  cudaStream_t st[kPoolStreams] = {};
  cudaEvent_t ev[kPoolStreams] = {};
};

StreamPool& stream_pool(int dev) {
  static StreamPool tab[64];
  static std::mutex mu;
  std::lock_guard<std::mutex> lk(mu);
  StreamPool& p = tab[dev & 63];
  if (!p.ok) {
    bool good = true;
    for (int i = 0; i < kPoolStreams && good; ++i)
      good = cudaStreamCreateWithFlags(&p.st[i], cudaStreamNonBlocking) == cudaSuccess &&
             cudaEventCreateWithFlags(&p.ev[i], cudaEventDisableTiming) == cudaSuccess;
    p.ok = good;
  }
  return p;
}

enum Phase { kResid, kCycle, kArnoldi, kDone };   // kCycle with Arnoldi step 0 where that is issued ahead

struct BatchItem {
  Solver s;
  Phase ph = kResid;
  int j = 0;            // next Arnoldi step
  bool first = true;    // the first residual also takes ||A||
  bool finish = false;  // cycle_finish + update to issue before the next residual
  cudaEvent_t ev = nullptr;
  Report* host = nullptr;   // pinned copy of the report
};

size_t batch_solve_bytes(const hpmxp_problem* probs, int count, int restart) {
  size_t b = 0;
  for (int q = 0; q < count; ++q) b += round_up<size_t>(solve_ws_bytes(probs[q].n, probs[q].nrhs, restart), 256);
  return b;
}
}  // namespace

size_t solve_batched_ws_bytes(const hpmxp_problem* probs, int count, int restart) {
  return batch_solve_bytes(probs, count, restart);
}

hpmxp_status solve_ir_batched(const hpmxp_problem* probs, int count, int prec, const hpmxp_ir_params& prm,
                              hpmxp_ir_info* info, void* ws, cudaStream_t caller) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return status_from_cuda(e);
  StreamPool& pool = stream_pool(dev);
  if (!pool.ok) return HPMXP_ECUDA;
  std::lock_guard<std::mutex> lk(pool.mu);   // one batched solve drives a device's pool at a time
  // pinned briefs and per-system events, kept by the calling thread
  struct HostSide {
    Report* pinned = nullptr;
    size_t cap = 0;
    std::vector<cudaEvent_t> ev;
    ~HostSide() {
      if (pinned) cudaFreeHost(pinned);
      for (cudaEvent_t x : ev) cudaEventDestroy(x);
    }
  };
  thread_local HostSide hs;
  const size_t need = (size_t)count;
  if (hs.cap < need) {
    if (hs.pinned) cudaFreeHost(hs.pinned);
    hs.pinned = nullptr;
    hs.cap = 0;
    if ((e = cudaMallocHost(&hs.pinned, sizeof(Report) * need)) != cudaSuccess) return status_from_cuda(e);
    hs.cap = need;
  }
  while ((int)hs.ev.size() < count) {
    cudaEvent_t x;
    if ((e = cudaEventCreateWithFlags(&x, cudaEventDisableTiming)) != cudaSuccess) return status_from_cuda(e);
    hs.ev.push_back(x);
  }
  std::vector<BatchItem> it((size_t)count);
  char* base = (char*)ws;
  for (int q = 0; q < count; ++q) {
    Solver& s = it[q].s;
    s.n = probs[q].n; s.K = (int)probs[q].nrhs; s.m = prm.restart;
    s.A = probs[q].A; s.lda = probs[q].lda;
    s.LU = (const uint16_t*)probs[q].LU; s.ldlu = probs[q].ldlu; s.fmt = fmt_of(prec);
    s.B = probs[q].b; s.ldb = probs[q].ldb; s.X = probs[q].x; s.ldx = probs[q].ldx;
    s.prm = prm;
    s.w = carve_solve(base, s.n, s.K, prm.restart);
    s.w.pdl = false;
    base += round_up<size_t>(s.w.bytes, 256);
    s.st = pool.st[q % kPoolStreams];
    it[q].ev = hs.ev[q];
    it[q].host = hs.pinned + q;
  }
  // fork from the caller's stream
  cudaEvent_t fork_ev = pool.ev[0];
  if ((e = cudaEventRecord(fork_ev, caller)) != cudaSuccess) return status_from_cuda(e);
  for (int i = 0; i < kPoolStreams && i < count; ++i)
    if ((e = cudaStreamWaitEvent(pool.st[i], fork_ev, 0)) != cudaSuccess) return status_from_cuda(e);
  for (int q = 0; q < count && e == cudaSuccess; ++q) {
    Solver& s = it[q].s;
    if ((e = s.setup()) == cudaSuccess) e = s.precond(s.B, s.ldb, s.X, s.ldx);   // x0 = U^{-1} L^{-1} b
  }
  auto any = [](const BatchItem& b, int Brief::*f) {
    for (int r = 0; r < b.s.K; ++r)
      if (b.host->brief[r].*f) return true;
    return false;
  };
  const bool ahead = !prof_on();
  int active = count;
  while (active > 0 && e == cudaSuccess) {
    // issue every active system's next phase
    for (int q = 0; q < count && e == cudaSuccess; ++q) {
      BatchItem& b = it[q];
      if (b.ph == kDone) continue;
      Solver& s = b.s;
      if (b.finish) {
        e = s.cycle_finish();
        b.finish = false;
      }
      if (e != cudaSuccess) break;
      bool unchecked = false;
      if (b.ph == kResid) {
        e = s.outer_check(b.first);
        unchecked = b.first && ahead;
        if (unchecked) b.ph = kCycle;   // what Solver::run issues ahead
        b.first = false;
      } else if (b.ph == kArnoldi) {
        e = s.arnoldi_step(b.j, false);
      }
      if (e == cudaSuccess && b.ph == kCycle) {
        e = s.cycle_start(unchecked);
        if (e == cudaSuccess && ahead) e = s.arnoldi_step(0, true);
      }
      if (e == cudaSuccess) e = cudaMemcpyAsync(b.host, s.w.report, s.report_bytes(), cudaMemcpyDeviceToHost, s.st);
      if (e == cudaSuccess) e = cudaEventRecord(b.ev, s.st);
    }
    if (e != cudaSuccess) break;
    // one decision point for the batch
    for (int q = 0; q < count && e == cudaSuccess; ++q) {
      BatchItem& b = it[q];
      if (b.ph == kDone) continue;
      if ((e = cudaEventSynchronize(b.ev)) != cudaSuccess) break;
      if (b.ph == kResid) {
        b.ph = any(b, &Brief::outer_active) ? kCycle : kDone;
      } else if (b.ph == kCycle) {
        if (!any(b, &Brief::outer_active)) {
          b.ph = kDone;
        } else if (any(b, &Brief::cycle_active) && b.s.m > (ahead ? 1 : 0)) {
          b.ph = kArnoldi;
          b.j = ahead ? 1 : 0;
        } else {
          b.finish = true;
          b.ph = kResid;
        }
      } else {
        b.j += 1;
        if (!(b.j < b.s.m && any(b, &Brief::cycle_active))) {
          b.finish = true;
          b.ph = kResid;
        }
      }
      if (b.ph == kDone) --active;
    }
  }
  // join back to the caller's stream
  for (int i = 0; i < kPoolStreams && i < count; ++i) {
    cudaEventRecord(pool.ev[i], pool.st[i]);
    cudaStreamWaitEvent(caller, pool.ev[i], 0);
  }
  if (e != cudaSuccess) return status_from_cuda(e);
  int worst = HPMXP_OK;
  int64_t off = 0;
  for (int q = 0; q < count; ++q) {
    BatchItem& b = it[q];
    // the status word came with the last report
    if (b.host->status && worst == HPMXP_OK) worst = status_from_word(b.host->status);
    for (int r = 0; r < b.s.K; ++r) {
      if (info) {
        info[off + r].iters = b.host->brief[r].iters;
        info[off + r].outer = b.host->brief[r].outer;
        info[off + r].scaled_resid = b.host->brief[r].sr;
        info[off + r].status = b.host->brief[r].status;
        info[off + r].reserved = 0;
      }
      if (b.host->brief[r].status != HPMXP_OK && worst == HPMXP_OK) worst = b.host->brief[r].status;
    }
    off += b.s.K;
  }
  return (hpmxp_status)worst;
}

hpmxp_status precond_apply(int64_t n, const void* LU, int64_t ldlu, int fmt, const double* v, int64_t ldv,
                           double* z, int64_t ldz, int64_t nrhs, int fp32, void* ws, cudaStream_t st,
                           const double* rs, const double* cs) {
  Solver s;
  s.n = n; s.K = (int)nrhs; s.m = 1;
  s.LU = (const uint16_t*)LU; s.ldlu = ldlu; s.fmt = fmt;
  s.rs = rs; s.cs = cs;
  hpmxp_ir_params_default(&s.prm);
  s.prm.precond_fp32 = fp32;
  s.w = carve_solve(ws, n, nrhs, 1);
  s.st = st;
  cudaError_t e = s.setup();
  if (e == cudaSuccess) e = s.precond(v, ldv, z, ldz);
  uint32_t word = 0;
  if (e == cudaSuccess) e = read_to_host(&word, s.w.status, 4, st);
  if (e != cudaSuccess) return status_from_cuda(e);
  return status_from_word(word);
}

// r = b - A x (fp64, the refinement's residual kernels), every column.  Ordered
// on the stream like the work it launches, not waited for, so a wait that runs out
// in the tensor-core product cannot be reported: the last pass makes it good.
hpmxp_status residual_vector(int64_t n, const double* A, int64_t lda, const double* x, int64_t ldx,
                             const double* b, int64_t ldb, int64_t nrhs, double* r, int64_t ldr, void* ws,
                             cudaStream_t st) {
  SolveWs w = carve_solve(ws, n, nrhs, 1);
  cudaError_t e = cudaMemsetAsync(w.status, 0, 4, st);
  if (e == cudaSuccess) e = residual(n, (int)nrhs, A, lda, x, ldx, b, ldb, r, ldr, 0, 0, w, st, {}, {}, true);
  return status_from_cuda(e);
}

hpmxp_status residual_check(int64_t n, const double* A, int64_t lda, const double* x, int64_t ldx,
                            const double* b, int64_t ldb, int64_t nrhs, double* out, void* ws, cudaStream_t st) {
  SolveWs w = carve_solve(ws, n, nrhs, 1);
  cudaError_t e = cudaMemsetAsync(w.st, 0, sizeof(RhsState) * kMaxK, st);
  if (e != cudaSuccess) return status_from_cuda(e);
  e = residual(n, (int)nrhs, A, lda, x, ldx, b, ldb, w.r, n, 2, 1, w, st);
  if (e != cudaSuccess) return status_from_cuda(e);
  std::vector<RhsState> hs(nrhs);
  e = read_to_host(hs.data(), w.st, sizeof(RhsState) * (size_t)nrhs, st);
  if (e != cudaSuccess) return status_from_cuda(e);
  for (int64_t r = 0; r < nrhs; ++r) {
    double rn, xn, bn, an;
    memcpy(&rn, &hs[r].rn_bits, 8); memcpy(&xn, &hs[r].xn_bits, 8);
    memcpy(&bn, &hs[r].bn_bits, 8); memcpy(&an, &hs[r].an_bits, 8);
    out[r] = rn / ((an * xn + bn) * ((double)n * 0x1p-53));
  }
  return HPMXP_OK;
}

}  // namespace hpmxp
