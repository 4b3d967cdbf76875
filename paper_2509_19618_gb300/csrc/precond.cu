// Preconditioner application z = U^{-1} L^{-1} v with the 16-bit factors (section
// "Algorithmic Framework": the factors as a left preconditioner) in T = float or
// double arithmetic, both sweeps in one cooperative launch.
//
// A sweep is a chain over block rows (128 rows in fp32, 64 in fp64) owned
// round-robin by the CTAs.  With the inverted diagonal block and the two blocks
// before the diagonal multiplied by it once per solve,
//   Linv_b = L_bb^{-1},  P0_b = Linv_b L(b, b-1),  P1_b = Linv_b L(b, b-2),
// a block's solution is
//   z_b = Linv_b (v_b - sum_{k <= b-3} L(b, k) z_k) - P1_b z_{b-2} - P0_b z_{b-1},
// so that the chain's step is one product by a block held in registers, and the
// rest of a block's work has two steps' time.  A CTA has two groups of 256
// threads: the chain group does that for its owned blocks, the update group
// subtracts L(b, k) z_k, k <= b-3, from all of them, its 16-bit tiles streamed
// ahead of z_k into a ring.  Blocks are published as tagged words ((value half |
// epoch << 32), one per fp32 and two per fp64 value), so that a reader's poll
// delivers the data; each group polls for itself, with bounded waits.  The
// backward sweep is the same over U with the blocks in reverse.  Every block
// takes its terms in one order, whatever the number of CTAs.
//
// Bound by the chain of 2 n / 128 steps (2 n / 64 in fp64): a product by P0 and a
// hand-off through L2, and for the update group one tile per step.  Traced at
// n = 8192, one right-hand side: 1.25 us a step, of which P0 0.25 and the
// hand-off 0.3; the update group needs 0.5 for a tile and 0.3 to receive.  In
// fp64 the fp64 unit's FMAs (two a clock and SM) take most of a step, from
// n = 16384 the tiles' count does.  One application, with one group per CTA
// and the whole block row on the chain before:
//   fp32  n = 1024: 35 -> 24.5 us   8192, 8 right-hand sides: 575 -> 450
//         n = 32768: 1430 -> 826    8192, one: 155
//   fp64  n = 4096, 2 right-hand sides: 858 -> 494   one: 352
#include "internal.h"

#include <algorithm>
#include <type_traits>

namespace hpmxp {
namespace {

template <class T> constexpr int kTB = sizeof(T) == 4 ? 128 : 64;   // rows of a block
constexpr int kGrp = 256;                                           // threads of a group
template <class T> constexpr int kSlots = sizeof(T) == 4 ? 2 : 4;   // tiles in the update group's ring

template <class T> __device__ inline T fma_t(T a, T b, T c);
template <> __device__ inline float fma_t<float>(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <> __device__ inline double fma_t<double>(double a, double b, double c) { return __fma_rn(a, b, c); }
// a 16-bit factor entry as T (exact either way; the fp64 one built with integer operations)
template <class T> __device__ inline T u16_to(uint16_t h, int fmt);
template <> __device__ inline float u16_to<float>(uint16_t h, int fmt) { return u16_to_f32(h, fmt); }
template <> __device__ inline double u16_to<double>(uint16_t h, int fmt) { return u16_to_f64(h, fmt); }

// Inverse of diagonal block c (c < nb) of the unit-lower L (which == 0) or of
// U (which == 1) in T arithmetic, from the 16-bit factors.  Output inv[(which *
// nb + c) * TB * TB + j * TB + i] = inverse(i, j).  A CTA makes 32 columns
// (grid z), one per lane: row by row, the finished row's term is added to the
// rows still open, which are dealt out to the warps and kept in registers, so
// that the FMAs between two barriers are independent.  Bound by the 128 steps'
// latency (fp32) and the fp64 unit, where a warp's FMA takes 64 clocks of its
// scheduler (fp64).  fp32 46 us at n = 1024 and 210 us at 32768; one thread per
// column, a chain of dependent FMAs on one SM per block, took 80 and 328 us.
constexpr int kInvCols = 32, kInvPitch = kInvCols + 1, kInvThreads = 256;
template <class T>
__device__ inline T quotient(T s, T d, T r);   // s / d with r = 1 / d
template <>
__device__ inline float quotient<float>(float s, float d, float r) { return __fdiv_rn(s, d); }
// One correction of s * r: the plain fp64 division costs about ten fp64 instructions.  Correctly
// rounded like it (while nothing underflows): d has at most 11 significant bits, so no quotient lies
// within 2^-12 of its last place of a midpoint, r is rounded once, the remainder is exact, and the
// corrected quotient before its rounding is off by about 2^-52 of that place.
template <>
__device__ inline double quotient<double>(double s, double d, double r) {
  const double q = s * r;
  const double x = __fma_rn(__fma_rn(-q, d, s), r, q);
  return isfinite(x) ? x : s / d;   // (a subnormal or infinite r)
}
template <class T>
__global__ void __launch_bounds__(kInvThreads) diag_inv_kernel(int64_t n, const uint16_t* __restrict__ LU, int64_t ld,
                                                               int fmt, bool vec, T* __restrict__ inv) {
  extern __shared__ __align__(16) unsigned char dsm_raw[];
  constexpr int TB = kTB<T>;
  T* t = reinterpret_cast<T*>(dsm_raw);   // t[k * TB + i] = block(i, k)
  T* x = t + TB * TB;                     // x[i * kInvPitch + lane] = inverse(i, j0 + lane) when row i is done
  T* dg = x + TB * kInvPitch;             // U's diagonal and its reciprocals
  T* rd = dg + TB;
  const int nb = (int)cdiv<int64_t>(n, TB);
  const int c = blockIdx.x, j0 = blockIdx.z * kInvCols, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool upper = blockIdx.y == 1;
  const int64_t base = (int64_t)c * TB;
  // the part of the block these columns need: rows and columns j0 .. 127 of L, 0 .. j0 + 31 of U
  const int lo = upper ? 0 : j0, hi = upper ? j0 + kInvCols : TB;
  // 16-byte loads, all in flight; single values where the columns are not 16-byte aligned and for the
  // last rows, which need not be padded (the last column's lie at the end of the array)
  uint4 raw[TB * TB / 8 / kInvThreads];
#pragma unroll
  for (int q = 0; q < TB * TB / 8 / kInvThreads; ++q) {
    const int chunk = tid + q * kInvThreads, k = chunk / (TB / 8), i = chunk % (TB / 8) * 8;
    raw[q] = make_uint4(0, 0, 0, 0);
    if (i + 8 > lo && i < hi && k >= lo && k < hi && base + k < n && base + i < n) {
      const uint16_t* src = LU + base + i + (base + k) * ld;
      if (vec && base + i + 8 <= n) {
        raw[q] = *reinterpret_cast<const uint4*>(src);
      } else {
        uint32_t w[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = base + i + e < n ? src[e] : 0;
        raw[q] = make_uint4(w[0] | w[1] << 16, w[2] | w[3] << 16, w[4] | w[5] << 16, w[6] | w[7] << 16);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < TB * TB / 8 / kInvThreads; ++q) {
    const int chunk = tid + q * kInvThreads, k = chunk / (TB / 8), i0 = chunk % (TB / 8) * 8;
    const uint32_t w[4] = {raw[q].x, raw[q].y, raw[q].z, raw[q].w};
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int i = i0 + e;
      const bool in = base + i < n && base + k < n;
      const T v = in ? u16_to<T>((uint16_t)(w[e >> 1] >> (16 * (e & 1))), fmt) : (T)0;
      // the strict triangle only, zeros elsewhere: a finished row's term is then a no-op for
      // the rows that are closed; U's diagonal apart
      t[k * TB + i] = (upper ? i < k : i > k) ? v : (T)0;
      if (upper && i == k) dg[i] = in ? v : (T)1;
    }
  }
  __syncthreads();
  if (upper && tid < TB) rd[tid] = (T)1 / dg[tid];
  __syncthreads();
  // rows warp + kWarps r of the lane's column, in registers
  constexpr int kWarps = kInvThreads / 32, kRows = TB / kWarps;
  T acc[kRows];
#pragma unroll
  for (int r = 0; r < kRows; ++r) acc[r] = warp + kWarps * r == j0 + lane ? (T)1 : (T)0;
#pragma unroll 1
  for (int step = 0; step < hi - lo; ++step) {
    const int k = upper ? hi - 1 - step : lo + step;
    // row k's warp finishes and publishes it (U: divided by the diagonal)
    if (warp == k % kWarps) {
      T xk = (T)0;
#pragma unroll
      for (int r = 0; r < kRows; ++r)
        if (k == warp + kWarps * r) xk = acc[r];
      x[k * kInvPitch + lane] = upper ? quotient<T>(xk, dg[k], rd[k]) : xk;
    }
    __syncthreads();
    const T xk = -x[k * kInvPitch + lane];
    const T* tk = t + k * TB + warp;
#pragma unroll
    for (int g = 0; g < kRows; g += 4) {   // four rows at a time, skipped when all are closed
      if (upper ? warp + kWarps * g >= k : warp + kWarps * (g + 3) <= k) continue;
#pragma unroll
      for (int r = g; r < g + 4; ++r) acc[r] = fma_t<T>(tk[kWarps * r], xk, acc[r]);
    }
  }
  for (int idx = tid; idx < TB * kInvCols; idx += kInvThreads) {   // rows outside lo .. hi - 1 are zero
    const int i = idx / kInvCols;
    if (i < lo || i >= hi) x[i * kInvPitch + idx % kInvCols] = (T)0;
  }
  __syncthreads();
  T* out = inv + ((int64_t)blockIdx.y * nb + c) * TB * TB + (int64_t)j0 * TB;
  for (int idx = tid; idx < TB * kInvCols; idx += kInvThreads)
    out[idx] = x[(idx % TB) * kInvPitch + idx / TB];
}

template <class T>
constexpr size_t diag_inv_smem() { return sizeof(T) * (kTB<T> * kTB<T> + kTB<T> * kInvPitch + 2 * kTB<T>); }
static_assert(diag_inv_smem<double>() <= 232448, "shared memory per CTA");


// Chain blocks P0 (grid y: 0 L, 2 U) and P1 (1 L, 3 U), once per solve: the
// inverted diagonal block of b times the factor tile next to the diagonal / the
// one after it, terms ascending.  out[(y * nb + b) * TB * TB + j * TB + i].  A
// CTA makes 32 columns (grid z); a warp stops at its rows' last nonzero of the
// triangular inverse, and the column groups take the row groups in opposite
// orders so that every scheduler has the same work.  Bound by the FMAs (fp64).
constexpr int kChainCols = 32;
template <class T>
__global__ void __launch_bounds__(256) chain_kernel(int64_t n, const uint16_t* __restrict__ LU, int64_t ld, int fmt,
                                                    const T* __restrict__ dinv, T* __restrict__ out) {
  constexpr int TB = kTB<T>, kRowGroups = TB / 32, kPer = TB / 8;   // columns per thread
  __shared__ __align__(16) T tile[TB][kChainCols];   // tile[t][j] = T(t, j0 + j)
  const int nb = (int)cdiv<int64_t>(n, TB);
  const int b = blockIdx.x, which = blockIdx.y >> 1, dist = 1 + (blockIdx.y & 1), j0 = blockIdx.z * kChainCols;
  const int nbr = which == 0 ? b - dist : b + dist;   // block column of the tile
  if (nbr < 0 || nbr >= nb) return;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int64_t r0 = (int64_t)b * TB, c0 = (int64_t)nbr * TB + j0;
  for (int idx = tid; idx < TB * kChainCols; idx += 256) {
    const int t = idx % TB, j = idx / TB;   // coalesced over t (column major source)
    const bool in = r0 + t < n && c0 + j < n;
    tile[t][j] = in ? u16_to<T>(LU[r0 + t + (c0 + j) * ld], fmt) : (T)0;
  }
  __syncthreads();
  const T* inv = dinv + ((int64_t)which * nb + b) * TB * TB;
  const int cg = warp / kRowGroups, rg = (cg & 1) ? kRowGroups - 1 - warp % kRowGroups : warp % kRowGroups;
  const int i = 32 * rg + (tid & 31), jh = cg * kPer;
  const int t0 = which == 0 ? 0 : 32 * rg, t1 = which == 0 ? 32 * rg + 32 : TB;
  T acc[kPer];
#pragma unroll
  for (int q = 0; q < kPer; ++q) acc[q] = (T)0;
#pragma unroll 4
  for (int t = t0; t < t1; ++t) {
    const T a = inv[(int64_t)t * TB + i];
#pragma unroll
    for (int q = 0; q < kPer; ++q) acc[q] = fma_t<T>(a, tile[t][jh + q], acc[q]);
  }
  T* o = out + ((int64_t)blockIdx.y * nb + b) * TB * TB;
#pragma unroll
  for (int q = 0; q < kPer; ++q) o[(int64_t)(j0 + jh + q) * TB + i] = acc[q];
}

// words of one published value
template <class T> constexpr int kWords = sizeof(T) / 4;

__device__ inline unsigned long long tag_word(uint32_t bits, int epoch) {
  return (unsigned long long)bits | ((unsigned long long)(unsigned)epoch << 32);
}
// N consecutive shared values, 16 bytes a load where N values are a multiple of
// that, 8 for two fp32 values
template <int N, class T>
__device__ inline void load16(T (&v)[N], const T* src) {
  if constexpr (N * sizeof(T) % 16 == 0) {
    using V = std::conditional_t<sizeof(T) == 4, float4, double2>;
#pragma unroll
    for (int k = 0; k < N; k += 16 / (int)sizeof(T)) {
      const V w = *reinterpret_cast<const V*>(src + k);
      v[k] = w.x, v[k + 1] = w.y;
      if constexpr (sizeof(T) == 4) v[k + 2] = w.z, v[k + 3] = w.w;
    }
  } else if constexpr (sizeof(T) == 4 && N == 2) {
    const float2 w = *reinterpret_cast<const float2*>(src);
    v[0] = w.x, v[1] = w.y;
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) v[k] = src[k];
  }
}
// N values of global memory, past L1
__device__ inline void load16g(float (&v)[4], const float* src) {
  const float4 w = __ldcg(reinterpret_cast<const float4*>(src));
  v[0] = w.x, v[1] = w.y, v[2] = w.z, v[3] = w.w;
}
__device__ inline void load16g(float (&v)[2], const float* src) {
  const float2 w = __ldcg(reinterpret_cast<const float2*>(src));
  v[0] = w.x, v[1] = w.y;
}
template <class T>
__device__ inline void load16g(T (&v)[1], const T* src) { v[0] = __ldcg(src); }
__device__ inline void cp_async16(uint32_t dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ inline void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ inline void group_sync(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kGrp) : "memory"); }
// barrier of the group; true for all of its threads when v is true for all
__device__ inline bool group_all(int id, bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(id), "n"(kGrp)
      : "memory");
  return r != 0;
}

// Shared memory, in T: the two blocks of the chain group (P1 optional: a CTA
// with many blocks and right-hand sides reads it from L2), the ring, the owned
// blocks' right-hand sides and the groups' vectors and partial sums.
template <class T>
struct Smem {
  static constexpr int TB = kTB<T>;
  static constexpr int HG = kGrp / TB, HC = TB / HG;               // chain group: column groups of a product, their width
  static constexpr int CG = kGrp / 32 * 64 / TB, CC = TB / CG;     // update group, likewise
  static size_t bytes(int nown, int K, bool p1) {
    return sizeof(T) * ((size_t)(p1 ? 2 : 1) * TB * TB + (size_t)nown * TB * K + (size_t)(HG + CG + 1) * TB * K) +
           sizeof(uint16_t) * kSlots<T> * TB * TB;
  }
};
constexpr size_t kMaxPrecondSmem = 226 * 1024;

template <int N> using Int = std::integral_constant<int, N>;

struct PrecondArgs {
  int64_t n;
  const uint16_t* LU; int64_t ld; int fmt;
  const void* dinv;
  const void* chain;
  const double* v; int64_t ldv;
  double* z; int64_t ldz;
  unsigned long long* pub;
  int epoch;
  int p1_smem;
  uint32_t* status;
  long long wait_polls;
  unsigned long long wait_ns;
  const double* rs;
  const double* cs;
  Gate gate;
};

template <class T, int K>
__global__ void __launch_bounds__(2 * kGrp) precond_kernel(PrecondArgs p) {
  using S = Smem<T>;
  constexpr int TB = S::TB, HG = S::HG, HC = S::HC, CG = S::CG, CC = S::CC, W = kWords<T>, NS = kSlots<T>;
  // Rows of a lane in the chain group's and the update group's products: a value of x read from
  // shared memory serves that many sums (fp32, bound by those reads; more right-hand sides leave
  // registers for two).  fp64 is bound by its FMAs and takes the least additions between lanes.
  constexpr int kR = sizeof(T) == 8 ? 1 : K <= 3 ? 4 : 2, kRB = sizeof(T) == 8 ? 2 : kR;
  constexpr int kQ = K * sizeof(T) <= 16 || (sizeof(T) == 8 && K <= 4) ? 4 : K % 2 == 0 || sizeof(T) == 8 ? 2 : 1;   // columns of a run
  constexpr int kUnroll = K * sizeof(T) <= 8 ? 4 : sizeof(T) == 4 || K == 2 ? 2 : 1;   // runs read ahead, against registers
  if (p.gate.closed()) return;
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ volatile int ready;   // owned blocks of the sweep whose updates are complete
  const int nb = (int)cdiv<int64_t>(p.n, TB);
  const int G = gridDim.x, me = blockIdx.x, tid = threadIdx.x, gt = tid % kGrp;
  const bool chain_group = tid < kGrp;
  const int bar = chain_group ? 1 : 2;
  const int nown = (nb - me + G - 1) / G;
  T* linv = reinterpret_cast<T*>(sm_raw);
  T* p1s = linv + TB * TB;
  uint16_t* tl = reinterpret_cast<uint16_t*>(p.p1_smem ? p1s + TB * TB : p1s);   // [NS][TB][TB], tl[j * TB + i]
  T* acc = reinterpret_cast<T*>(tl + NS * TB * TB);   // [nown][TB][K]
  T* zA = acc + (size_t)nown * TB * K;                // chain group: a received block, partial sums
  T* partA = zA + TB * K;
  T* zB = partA + (HG - 1) * TB * K;                  // update group
  T* partB = zB + TB * K;
  for (int o = 0; o < nown; ++o)
    for (int t = tid; t < TB * K; t += 2 * kGrp) {
      const int ii = t % TB, r = t / TB;
      const int64_t i = (int64_t)(me + o * G) * TB + ii;
      // balanced factors (LU of diag(rs) A diag(cs)): M^{-1} v = diag(cs) U^{-1} L^{-1} diag(rs) v;
      // rs and cs are powers of two, so the scalings are exact
      acc[((size_t)o * TB + ii) * K + r] = i < p.n ? (T)(p.rs ? p.v[i + r * p.ldv] * p.rs[i] : p.v[i + r * p.ldv]) : (T)0;
    }

  // A published block is read in two steps.  peek: the group's threads load the block's tagged
  // words, which they use only later, so that the loads' latency passes beside other work;
  // take: words that were not there yet are polled, the values go to dst.  take returns false for
  // the whole group when a wait ran out (the timeout bit is set) and ends with the group's barrier.
  constexpr int kPer = (TB * K + kGrp - 1) / kGrp;   // values per thread
  unsigned long long peeked[kPer][W];
  auto word_at = [&](const unsigned long long* src, int b, int t, int h) {
    unsigned long long word;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(word)
                 : "l"(src + ((size_t)b * TB * K + t) * W + h) : "memory");
    return word;
  };
  auto peek = [&](const unsigned long long* src, int b) {
#pragma unroll
    for (int e = 0; e < kPer; ++e)
#pragma unroll
      for (int h = 0; h < W; ++h)
        if (gt + e * kGrp < TB * K) peeked[e][h] = word_at(src, b, gt + e * kGrp, h);
  };
  auto take = [&](const unsigned long long* src, int b, T* dst) {
    bool got = true;
#pragma unroll
    for (int e = 0; e < kPer; ++e) {
      const int t = gt + e * kGrp;
      if (t < TB * K) {
        uint32_t bits[W];
#pragma unroll
        for (int h = 0; h < W; ++h) {
          unsigned long long word = peeked[e][h], t0 = 0;
          for (long long it = 0; got && (int)(word >> 32) != p.epoch; ++it) {
            if (it == 0) t0 = global_ns();
            if (it >= p.wait_polls || ((it & 63) == 63 && global_ns() - t0 > p.wait_ns)) {
              atomicOr(p.status, kErrTimeout);
              got = false;
            }
            word = word_at(src, b, t, h);
          }
          bits[h] = (uint32_t)word;
        }
        if constexpr (W == 1) dst[t] = __uint_as_float(bits[0]);
        else dst[t] = __hiloint2double((int)bits[0], (int)bits[1]);
      }
    }
    return group_all(bar, got);
  };

  for (int sweep = 0; sweep < 2; ++sweep) {   // forward over L, backward over U
    // positions 0 .. nb-1 of the chain; this CTA owns positions p0, p0 + G, ...
    const int p0 = sweep == 0 ? me : nb - 1 - (me + (nown - 1) * G);
    auto block_at = [&](int pos) { return sweep == 0 ? pos : nb - 1 - pos; };
    auto acc_of = [&](int o) { return acc + (size_t)(sweep == 0 ? o : nown - 1 - o) * TB * K; };
    unsigned long long* pub = p.pub + (size_t)sweep * nb * TB * K * W;
    // every CTA is resident: the next kernel's may wait beside them, but not for both sweeps, since they
    // take that long room from other streams' kernels (n = 8192, four right-hand sides, solved by two
    // threads on their own streams: 2430 us a solve from the start on, 2280 from here; alone 3445 either way)
    if (sweep == 1) pdl_trigger();
    if (tid == 0) ready = 0;
    __syncthreads();   // acc: the sweep's right-hand sides
    if (chain_group) {
      // a product by a block: a warp has 32 rows and the columns of group h, a lane kR rows (one
      // load per column) and every kR-th run of kQ columns
      const int lane = gt & 31, rb = (gt >> 5) % (TB / 32), h = (gt >> 5) / (TB / 32), cl = lane / (32 / kR);
      const int rowR = 32 * rb + kR * (lane % (32 / kR)), ii = rowR + cl;   // ii: the row whose sum the lane ends up with
      auto col_of = [&](int q) { return h * HC + (q * kR + cl) * kQ; };
      T pr0[HC / kR][kR];
      bool ok = true;
      for (int o = 0; o < nown && ok; ++o) {
        const int pos = p0 + o * G, b = block_at(pos);
        const T* dv = static_cast<const T*>(p.dinv) + ((int64_t)sweep * nb + b) * TB * TB;
        const T* c0 = static_cast<const T*>(p.chain) + ((int64_t)(2 * sweep) * nb + b) * TB * TB;
        const T* c1 = c0 + (int64_t)nb * TB * TB;
        for (int q = gt * 16 / (int)sizeof(T); q < TB * TB; q += kGrp * 16 / (int)sizeof(T)) {
          cp_async16((uint32_t)__cvta_generic_to_shared(linv + q), dv + q, 16);
          if (p.p1_smem && pos >= 2) cp_async16((uint32_t)__cvta_generic_to_shared(p1s + q), c1 + q, 16);
        }
        cp_async_commit();
        if (pos >= 1) {
#pragma unroll
          for (int q = 0; q < HC / kR; ++q) load16g(pr0[q], c0 + (col_of(q / kQ) + q % kQ) * TB + rowR);
        }
        // this thread's part of M x: the sums of its kR rows over its columns, then over the
        // column lanes; s is row ii's.  get(q, k, m): the rows of the lane's column k of its q-th run
        auto product = [&](auto unroll, auto get, const T* x, T (&s)[K]) {
          constexpr int kU = decltype(unroll)::value;
          T u[kR][K];
#pragma unroll
          for (int i = 0; i < kR; ++i)
#pragma unroll
            for (int r = 0; r < K; ++r) u[i][r] = (T)0;
#pragma unroll(kU)
          for (int q = 0; q < HC / kR / kQ; ++q) {
            T xv[kQ * K];
            load16(xv, x + col_of(q) * K);
#pragma unroll
            for (int k = 0; k < kQ; ++k) {
              T m[kR];
              get(q, k, m);
#pragma unroll
              for (int i = 0; i < kR; ++i)
#pragma unroll
                for (int r = 0; r < K; ++r) u[i][r] = fma_t<T>(m[i], xv[k * K + r], u[i][r]);
            }
          }
#pragma unroll
          for (int r = 0; r < K; ++r) {
            if constexpr (kR == 4) {   // upper half of the rows to the upper lanes
              const bool up = cl & 2;
#pragma unroll
              for (int i = 0; i < 2; ++i)
                u[i][r] = (up ? u[2 + i][r] : u[i][r]) + __shfl_xor_sync(0xffffffffu, up ? u[i][r] : u[2 + i][r], 16);
            }
            if constexpr (kR >= 2) {
              const bool up = cl & 1;
              u[0][r] = (up ? u[1][r] : u[0][r]) + __shfl_xor_sync(0xffffffffu, up ? u[0][r] : u[1][r], 32 / kR);
            }
            s[r] = u[0][r];
          }
        };
        auto rows_of = [&](const T* M) {
          return [=](int q, int k, T (&m)[kR]) { load16(m, M + (col_of(q) + k) * TB + rowR); };
        };
        auto rows_of_global = [&](const T* M) {
          return [=](int q, int k, T (&m)[kR]) { load16g(m, M + (col_of(q) + k) * TB + rowR); };
        };
        // the column groups' parts, summed in order by the threads with h == 0
        auto combine = [&](T (&s)[K]) {
          if (h > 0) {
#pragma unroll
            for (int r = 0; r < K; ++r) partA[((h - 1) * TB + ii) * K + r] = s[r];
          }
          group_sync(bar);
          if (h == 0) {
#pragma unroll
            for (int g = 1; g < HG; ++g)
#pragma unroll
              for (int r = 0; r < K; ++r) s[r] += partA[((g - 1) * TB + ii) * K + r];
          }
        };
        T* a = acc_of(o);
        if (pos >= 3) {   // every term but the last two has been subtracted
          unsigned long long t0 = 0;
          for (long long it = 0; ok && ready <= o; ++it) {
            if (it == 0) t0 = global_ns();
            if (it >= p.wait_polls || ((it & 63) == 63 && global_ns() - t0 > p.wait_ns)) {
              atomicOr(p.status, kErrTimeout);
              ok = false;
            }
          }
          __threadfence_block();
        }
        cp_async_wait<0>();
        ok = group_all(bar, ok);
        if (!ok) break;
        T y[K], s[K];
        if (pos >= 2) peek(pub, block_at(pos - 2));
        product(Int<kUnroll>{}, rows_of(linv), a, y);
        combine(y);
        if (pos >= 2) {
          ok = take(pub, block_at(pos - 2), zA);
          if (!ok) break;
          if (p.p1_smem) product(Int<kUnroll>{}, rows_of(p1s), zA, s);
          else product(Int<kUnroll>{}, rows_of_global(c1), zA, s);
          peek(pub, block_at(pos - 1));
          combine(s);
#pragma unroll
          for (int r = 0; r < K; ++r) y[r] -= s[r];
        }
        if (pos >= 1) {
          if (pos == 1) peek(pub, block_at(0));
          ok = take(pub, block_at(pos - 1), zA);
          if (!ok) break;
          product(Int<HC / kR / kQ>{}, [&](int q, int k, T (&m)[kR]) {
#pragma unroll
            for (int i = 0; i < kR; ++i) m[i] = pr0[q * kQ + k][i];
          }, zA, s);
          combine(s);
#pragma unroll
          for (int r = 0; r < K; ++r) y[r] -= s[r];
        }
        if (h == 0) {
          unsigned long long* wd = pub + ((size_t)b * TB + ii) * K * W;
#pragma unroll
          for (int r = 0; r < K; ++r) {
            if constexpr (W == 1) {
              asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(wd + r),
                           "l"(tag_word(__float_as_uint(y[r]), p.epoch)) : "memory");
            } else {
              asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(wd + 2 * r),
                           "l"(tag_word((uint32_t)__double2hiint(y[r]), p.epoch)) : "memory");
              asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(wd + 2 * r + 1),
                           "l"(tag_word((uint32_t)__double2loint(y[r]), p.epoch)) : "memory");
            }
          }
          const int64_t i = (int64_t)b * TB + ii;
#pragma unroll
          for (int r = 0; r < K; ++r) {
            a[ii * K + r] = y[r];   // the backward sweep's right-hand side
            if (sweep == 1 && i < p.n) p.z[i + r * p.ldz] = p.cs ? (double)y[r] * p.cs[i] : (double)y[r];
          }
        }
        group_sync(bar);   // linv, p1s and partA are free
      }
      cp_async_wait<0>();
    } else {
      // pairs (c, o): position c's block updates owned position p0 + o G >= c + 3, c ascending
      const int last = p0 + (nown - 1) * G;
      auto first_o = [&](int c) { const int d = c + 3 - p0; return d <= 0 ? 0 : (d + G - 1) / G; };
      int fc = 0, fo = first_o(0), slot_f = 0;   // the next pair to fetch
      auto fetch = [&]() {
        if (fc + 3 <= last) {
          // 8 rows of a column per copy, zero outside the matrix
          constexpr int kRowPieces = TB / 8, kStep = kGrp / kRowPieces;
          const int ii = gt % kRowPieces * 8, jj = gt / kRowPieces;
          const int64_t i = (int64_t)block_at(p0 + fo * G) * TB + ii, j = (int64_t)block_at(fc) * TB + jj;
          const int bytes = i < p.n ? (int)min((int64_t)16, (p.n - i) * 2) : 0;
          const int cols = (int)min((int64_t)TB, p.n - j);   // copies with q * kStep < cols have data
          const uint16_t* src = p.LU + i + j * p.ld;
          const uint32_t dst = (uint32_t)__cvta_generic_to_shared(tl + (size_t)slot_f * TB * TB + jj * TB + ii);
#pragma unroll
          for (int q = 0; q < TB / kStep; ++q) {
            const int by = q * kStep < cols ? bytes : 0;
            cp_async16(dst + q * kStep * TB * 2, by ? src + (int64_t)q * kStep * p.ld : p.LU, by);
          }
          if (++fo >= nown) fo = first_o(++fc);
        }
        cp_async_commit();
        slot_f = slot_f + 1 == NS ? 0 : slot_f + 1;
      };
#pragma unroll
      for (int k = 0; k < NS; ++k) fetch();
      // a warp has 64 rows and the columns of group cg, a lane kRB rows and every
      // second run of kQ columns where it has four rows
      constexpr int CL = kRB / 2;
      const int lane = gt & 31, cl = lane / (32 / CL), cg = (gt >> 5) / (TB / 64);
      const int rowR = 64 * ((gt >> 5) % (TB / 64)) + kRB * (lane % (32 / CL));
      int slot = 0;
      bool ok = true;
      if (last >= 3) peek(pub, block_at(0));
      for (int c = 0; c + 3 <= last && ok; ++c) {
        cp_async_wait<NS - 1>();   // the first pair's tile; take's barrier makes it everyone's
        ok = take(pub, block_at(c), zB);
        if (!ok) break;
        if (c + 4 <= last) peek(pub, block_at(c + 1));
        for (int o = first_o(c), o0 = o; o < nown; ++o) {
          if (o > o0) {
            cp_async_wait<NS - 1>();
            group_sync(bar);
          }
          const uint16_t* tw = tl + (size_t)slot * TB * TB + rowR;
          T s[kRB][K];
#pragma unroll
          for (int i = 0; i < kRB; ++i)
#pragma unroll
            for (int r = 0; r < K; ++r) s[i][r] = (T)0;
          auto tile_product = [&](int fmt) {
#pragma unroll(kUnroll)
            for (int q = 0; q < CC / CL / kQ; ++q) {
              const int col = cg * CC + (q * CL + cl) * kQ;
              T xv[kQ * K];
              load16(xv, zB + col * K);
#pragma unroll
              for (int k = 0; k < kQ; ++k) {
                uint32_t w[kRB / 2];
                const uint32_t* src = reinterpret_cast<const uint32_t*>(tw + (col + k) * TB);
                if constexpr (kRB == 4) {
                  const uint2 v = *reinterpret_cast<const uint2*>(src);
                  w[0] = v.x, w[1] = v.y;
                } else {
                  w[0] = *src;
                }
#pragma unroll
                for (int i = 0; i < kRB; ++i) {
                  const T t = u16_to<T>((uint16_t)(w[i / 2] >> 16 * (i % 2)), fmt);
#pragma unroll
                  for (int r = 0; r < K; ++r) s[i][r] = fma_t<T>(t, xv[k * K + r], s[i][r]);
                }
              }
            }
          };
          if (p.fmt == kBF16) tile_product(kBF16);
          else tile_product(kFP16);
          // the sums of two column lanes: each keeps two of the four rows
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int r = 0; r < K; ++r) {
              T v = s[i][r];
              if constexpr (kRB == 4)
                v = (cl ? s[2 + i][r] : s[i][r]) + __shfl_xor_sync(0xffffffffu, cl ? s[i][r] : s[2 + i][r], 16);
              partB[(cg * TB + rowR + 2 * cl + i) * K + r] = v;
            }
          group_sync(bar);   // the tile has been read, the parts are there
          slot = slot + 1 == NS ? 0 : slot + 1;
          T* a = acc_of(o);
#pragma unroll
          for (int e = 0; e < (TB * K + kGrp - 1) / kGrp; ++e) {   // the parts, column groups in order
            const int t = gt + e * kGrp;
            if (t < TB * K) {
              T sum = partB[t];
#pragma unroll
              for (int g = 1; g < CG; ++g) sum += partB[g * TB * K + t];
              a[t] -= sum;
            }
          }
          if (p0 + o * G == c + 3) {   // complete but for the chain's two terms
            group_sync(bar);
            if (gt == 0) {
              __threadfence_block();
              ready = o + 1;
            }
          }
          fetch();
        }
      }
      cp_async_wait<0>();
    }
    __syncthreads();
  }
}

template <class T>
size_t precond_smem(int64_t n, int K, int G, bool p1) {
  return Smem<T>::bytes(cdiv((int)cdiv<int64_t>(n, kTB<T>), G), K, p1);
}

template <class T, int K>
cudaError_t launch_k(const PrecondArgs& args, const PrecondPlan& plan, cudaStream_t st) {
  auto kern = precond_kernel<T, K>;
  // one value for every call: concurrent solves on other threads set the same cap
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxPrecondSmem);
  if (e != cudaSuccess) return e;
  PrecondArgs a = args;
  void* ptrs[] = {&a};
  return cudaLaunchCooperativeKernel((const void*)kern, dim3(plan.ctas), dim3(2 * kGrp), ptrs, plan.smem, st);
}

template <class T>
cudaError_t launch(int K, const PrecondArgs& a, const PrecondPlan& plan, cudaStream_t st) {
  switch (K) {
    case 1: return launch_k<T, 1>(a, plan, st);
    case 2: return launch_k<T, 2>(a, plan, st);
    case 3: return launch_k<T, 3>(a, plan, st);
    case 4: return launch_k<T, 4>(a, plan, st);
    case 5: return launch_k<T, 5>(a, plan, st);
    case 6: return launch_k<T, 6>(a, plan, st);
    case 7: return launch_k<T, 7>(a, plan, st);
    default: return launch_k<T, 8>(a, plan, st);
  }
}

bool columns_aligned(const uint16_t* LU, int64_t ld) { return ld % 8 == 0 && reinterpret_cast<uintptr_t>(LU) % 16 == 0; }

template <class T>
cudaError_t setup(int64_t n, const uint16_t* LU, int64_t ld, int fmt, void* dinv, void* chain, cudaStream_t st) {
  constexpr size_t ism = diag_inv_smem<T>();
  cudaError_t e = cudaFuncSetAttribute(diag_inv_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ism);
  if (e != cudaSuccess) return e;
  const unsigned nb = (unsigned)cdiv<int64_t>(n, kTB<T>);
  diag_inv_kernel<T><<<dim3(nb, 2, kTB<T> / kInvCols), kInvThreads, ism, st>>>(n, LU, ld, fmt, columns_aligned(LU, ld), (T*)dinv);
  chain_kernel<T><<<dim3(nb, 4, kTB<T> / kChainCols), 256, 0, st>>>(n, LU, ld, fmt, (const T*)dinv, (T*)chain);
  count_launches(2);
  return cudaGetLastError();
}

}  // namespace

size_t precond_inverse_bytes(int64_t n) {   // fp32: 128-row blocks, fp64: 64-row blocks
  return sizeof(float) * 2 * round_up<int64_t>(n, 128) * 128;
}
size_t precond_chain_bytes(int64_t n) { return 2 * precond_inverse_bytes(n); }
// tagged words of both sweeps, sized for fp64 values (two words each)
size_t precond_pub_bytes(int64_t n, int64_t K) {
  return sizeof(unsigned long long) * 2 * 2 * round_up<int64_t>(n, 128) * K;
}

bool precond_plan(int64_t n, int K, bool fp32, int sms, int budget, PrecondPlan* plan) {
  // one CTA per SM at most: a cooperative launch keeps all of them resident
  const int nb = (int)cdiv<int64_t>(n, fp32 ? kTB<float> : kTB<double>);
  // one CTA per owned share of block rows; an SM budget takes fewer CTAs as
  // long as their shares still fit in shared memory
  const int gmax = std::max(1, std::min(nb, sms));
  int G = std::max(1, std::min(gmax, budget > 0 ? budget : gmax));
  auto bytes = [&](int g, bool p1) {
    return fp32 ? precond_smem<float>(n, K, g, p1) : precond_smem<double>(n, K, g, p1);
  };
  while (G < gmax && bytes(G, false) > kMaxPrecondSmem) ++G;
  plan->ctas = G;
  plan->p1_smem = bytes(G, true) <= kMaxPrecondSmem;
  plan->smem = bytes(G, plan->p1_smem);
  return plan->smem <= kMaxPrecondSmem;
}

cudaError_t precond_setup(int64_t n, const uint16_t* LU, int64_t ld, int fmt, bool fp32, void* dinv, void* chain,
                          cudaStream_t st) {
  // the update group's tiles are copied 16 bytes at a time; one block needs none
  if (n > 128 && !columns_aligned(LU, ld)) return cudaErrorInvalidValue;
  return fp32 ? setup<float>(n, LU, ld, fmt, dinv, chain, st) : setup<double>(n, LU, ld, fmt, dinv, chain, st);
}

cudaError_t precond_launch(const PrecondPlan& plan, bool fp32, int K, int64_t n, const uint16_t* LU, int64_t ld,
                           int fmt, const void* dinv, const void* chain, const double* v, int64_t ldv, double* z,
                           int64_t ldz, void* pub, int epoch, uint32_t* status, const double* rs, const double* cs,
                           cudaStream_t st, Gate gate) {
  const WaitBudget wb = wait_budget();
  const PrecondArgs a{n, LU, ld, fmt, dinv, chain, v, ldv, z, ldz, (unsigned long long*)pub, epoch,
                      plan.p1_smem ? 1 : 0, status, wb.polls, wb.ns, rs, cs, gate};
  return fp32 ? launch<float>(K, a, plan, st) : launch<double>(K, a, plan, st);
}

}  // namespace hpmxp
