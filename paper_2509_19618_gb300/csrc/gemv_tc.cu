// fp64 products A X of the refinement (section "Algorithmic Framework": the
// residual and the Arnoldi products in 64-bit precision) on the tensor cores.
//
// GB300's fp64 unit does two FMAs per clock and SM: n^2 K of them are what
// bounds the plain kernel (gemv_partial_kernel in ir.cu), 1.3 times the time of
// reading A for one right-hand side and ten times for eight.  Here the
// products are formed exactly from 8-bit digits instead (error-free splitting
// into slices whose products a matrix unit accumulates exactly: Ozaki, Ogita,
// Oishi and Rump, Numerical Algorithms 59, 2012):
//   - Column j of A and X is scaled by 2^e_j (e_j the largest exponent of x_j
//     over the right-hand sides, each right-hand side normalised by its own
//     2^f_r), so that A's entries carry the size of their products.
//   - Row i's scaled entries become 64-bit magnitudes below 2^(E + 1) of a
//     running exponent E, cut into eight 8-bit digits d_s with the entry's sign;
//     X's scaled values become 63-bit integers in eight signed 8-bit digits t_u.
//     Digits are exact in fp16.
//   - tcgen05 accumulates D_w = sum_{s+u=w} d_s t_u, w = 0 .. 7, over 64
//     columns: integers below 8 * 64 * 255 * 128 < 2^24, so every fp32 sum is
//     exact.
//   - D is added to 64-bit integers per row, right-hand side and half of the
//     weights; they become fp64 once per work unit.
// What is lost, against M_i = the largest |a_ij| 2^e_j met in the row's work unit
// (2^E <= 4 M_i): the bits of an entry below 2^(E - 63), none of one within 2^8
// of M_i; the bits of x_jr below 2^(e_j - 64), none of one within 2^10 of the
// largest x in its column; and the digit pairs with s + u > 7, at most 7 * 2^-64
// times 2^(E + 1).  Per column that is at most 2^-57 M_i, which is 2^-56 of the
// row's largest product for one right-hand side and, since E follows columns whose
// x_jr differ by 2^6 at most, 2^-50 of a side's own largest for several; the signs
// differ from column to column.  The plain kernel rounds every partial sum at
// 2^-53.  With seven digits on both sides a Gaussian A with a dominant diagonal was
// 1.5 to 2.3 times less accurate than the plain kernel (rms, n = 2048, two
// right-hand sides), rows whose largest products cancel 16 to 21 times; with eight
// digits the errors are 0.006 and 0.08 of the plain kernel's.
//
// An entry above 2^E (a diagonally dominant row's diagonal; a non-finite
// entry, whose exponent exceeds every E in use) has no digits: its product is
// added by fp64 FMAs from A and X, and E is raised after the third one of a
// row.  E follows columns that matter to every right-hand side (x_jr within
// 2^6 of the column's largest for all r); with hardly any such column, and in
// blocks with a non-finite x or an E at the ends of fp64's range, all products
// are fp64 FMAs, taken from the same stages (a second, direct read of A made
// matrices with zero blocks, whose rows have no E there, and unlike right-hand
// sides up to 2 times slower than gemv_partial_kernel).  Zero entries are skipped:
// n = 16384, four right-hand sides, lower triangular 2740 -> 440 us, unlike
// right-hand sides 2350 -> 1800 (the FMA kernel 1755).
//
// Layout: a CTA takes 512 rows, four groups of 128 threads (thread = row, TMEM
// lane), by 64-column blocks.  A's columns come by TMA (16 columns x 128 rows per
// box) into two stages per group, each refilled by a thread of the group after
// the group barrier that follows its last use; X's digits, made once per call by
// digit_kernel in the swizzled layout of the MMA's B operand, come into three
// buffers that the groups share.  A thread cuts its row's digits with integer
// instructions and stores them to TMEM (the MMA's A operand).  Slice s adds to D's
// columns 8 (s + u) + r of the block's 64.  Bound by the integer pipe (half the
// issue rate, about 18 of 36 instructions per entry) and the group's barriers: 425 us
// at n = 16384 with four right-hand sides, 1.46 ms at 32768 with one (5.9 TB/s of A),
// against 1.76 and 1.78 ms of fp64 FMAs.  (432 and 1.49 with seven digits and all MMAs
// issued on one scheduler, 458 and 1.58 with eight.)
#include "tcgen05.h"

#include <cuda_fp16.h>

#include <limits.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

namespace hpmxp {
namespace {

constexpr int kRowsT = 128;                  // rows of a group
constexpr int kBlk = 64;                     // columns of a block (exactness: see above)
constexpr int kGroups = 4;
constexpr int kTileRows = kGroups * kRowsT;
constexpr int kThr = kTileRows;
constexpr int kSlices = 8;
constexpr int kDig = kSlices * 1024;         // bytes of a block's X digits: 8 groups of 8 rows x 128 bytes
constexpr int kExpW = 2 * kBlk + 4;          // a block's column exponents (all, and of robust columns) and flag
constexpr int kExp = kExpW * 4;              // in bytes, whole 16-byte pieces
constexpr int kBBufs = 3;                    // digit buffers, a zero group of 8 rows before each
constexpr int kBArea = kBBufs * (kSlices + 1) * 1024;
constexpr int kCols = 16;                    // columns of a ring stage (one MMA's depth)
constexpr int kStage = kCols * kRowsT * 8;
constexpr int kStages = 2;                   // per group
constexpr int kTmA = 64, kTmD = 256;         // TMEM columns: group g's digits at 64 g, its D at 256 + 64 g
constexpr int kNoExp = -400;                 // exponent of a column whose x is zero, the least one kept
// E's range: below it zero and subnormal entries would get digits, above it a
// non-finite entry (exponent 2047) in a column of exponent kNoExp would not exceed it
constexpr int kMinE = 64, kMaxE = 2047 + kNoExp - 1;
static_assert((long long)kSlices * kBlk * 255 * 128 < (1 << 24), "exact fp32 sums");
constexpr int kBars = 2 * kBBufs + kGroups * kStages + 2 * kGroups;

template <int K>
constexpr size_t gemv_smem() {
  return 1024 + kBArea + (size_t)kGroups * kStages * kStage + (size_t)2 * K * kTileRows * 8 + kBBufs * kExp + 8 * kBars + 16;
}
static_assert(gemv_smem<8>() <= 232448, "shared memory per CTA");

// --- X's digits ------------------------------------------------------------

// f_r: 2^f_r > max_j |x_jr| (one CTA per right-hand side), or kOut where r is
// zero or not live: such a column takes no part in the column exponents, or it
// would decide how the others' products are formed (a zero one would send them
// all to fp64 FMAs, 8192 x 8: 1078 us instead of 157; one whose cycle has ended
// is unwritten workspace).
constexpr int kOut = 4096;
__global__ void __launch_bounds__(1024) xscale_kernel(int64_t n, const double* __restrict__ X, int64_t ldx,
                                                      int* __restrict__ fr, Gate gate, Gate live) {
  __shared__ int sh[32];
  pdl_wait();
  if (gate.closed()) return;
  pdl_trigger();
  const double* x = X + blockIdx.x * ldx;
  int m = 0;
  if (!live.flag || live.flag[(size_t)blockIdx.x * live.stride])
    for (int64_t j = threadIdx.x; j < n; j += 1024) {
      const double v = x[j];
      m = max(m, (__double2hiint(v) & 0x7fffffff) | (__double2loint(v) != 0));
    }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = __reduce_max_sync(0xffffffffu, sh[threadIdx.x]);
    if (threadIdx.x == 0) {
      fr[blockIdx.x] = m ? (m >> 20) - 1022 : kOut;
      if (blockIdx.x == 0) fr[8] = 0;   // digit_kernel counts the columns that are not robust
    }
  }
}

// Block b's digits (the swizzled K-major image of the B operand: row 8 u + r,
// column j), column exponents (times 2^20)
// and flag (1: an x that is not finite or too small for them).
__global__ void __launch_bounds__(512) digit_kernel(int64_t n, int K, const double* __restrict__ X, int64_t ldx,
                                                    int* __restrict__ fr, uint8_t* __restrict__ dig,
                                                    int* __restrict__ ex, Gate gate) {
  __shared__ int es[8][kBlk];
  __shared__ int bad;
  const int jl = threadIdx.x & (kBlk - 1), r = threadIdx.x / kBlk;
  const int64_t j = (int64_t)blockIdx.x * kBlk + jl;
  if (threadIdx.x == 0) bad = 0;
  pdl_wait();
  if (gate.closed()) return;
  pdl_trigger();
  double v = 0.0;
  const int f = r < K ? fr[r] : kOut;
  const bool skip = f == kOut;
  if (!skip && j < n) v = X[j + r * ldx];
  const bool fin = isfinite(v);
  if (!fin) v = 0.0;
  const int ev = v == 0.0 ? kNoExp : ilogb(v) + 1 - f;   // |v| 2^-f < 2^ev
  const int e = max(ev, kNoExp);
  es[r][jl] = skip ? INT_MIN : e;
  __syncthreads();
  if (!fin || ev < kNoExp) bad = 1;
  int em = kNoExp;
  for (int k = 0; k < K; ++k) em = max(em, es[k][jl]);
  bool robust = true;   // every right-hand side has a sizeable x in this column (or none has any)
  for (int k = 0; k < K; ++k) robust = robust && (es[k][jl] == INT_MIN || es[k][jl] >= em - 6);
  long long q = em == kNoExp ? 0 : llrint(scalbn(v, 63 - f - em));
  uint8_t* out = dig + (size_t)blockIdx.x * kDig + r * 128 + (((jl >> 3) ^ r) << 4) + (jl & 7) * 2;
#pragma unroll
  for (int u = kSlices - 1; u >= 0; --u) {
    const int d = u ? (int)((q + 128) & 255) - 128 : (int)q;
    q = (q - d) >> 8;
    *reinterpret_cast<__half*>(out + u * 1024) = __int2half_rn(d);
  }
  if (r == 0) {
    ex[(size_t)blockIdx.x * kExpW + jl] = em * (1 << 20);
    ex[(size_t)blockIdx.x * kExpW + kBlk + jl] = (robust ? em : kNoExp) * (1 << 20);
  }
  const int odd = __syncthreads_count(r == 0 && !robust);
  if (threadIdx.x == 0) {
    ex[(size_t)blockIdx.x * kExpW + 2 * kBlk] = bad;
    if (odd) atomicAdd(fr + 8, odd);
  }
}

// --- the product -----------------------------------------------------------

__device__ __forceinline__ void group_barrier(int g) {
  asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "n"(kRowsT) : "memory");
}
// `bytes` (a multiple of 16) from global to shared memory, completing on bar
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void tma_load_2d_stream(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t bar,
                                                   uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], "
      "[%4], %5;" ::"r"(dst),
      "l"((uint64_t)tm), "r"(x), "r"(y), "r"(bar), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t t, const uint32_t (&v)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(t), "r"(v[0]), "r"(v[1]),
               "r"(v[2]), "r"(v[3])
               : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t t, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(t));
}
// D += A B with A in tensor memory
__device__ __forceinline__ void tc_mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d), "r"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ int mad(int x, int y, int z) {
  int r;
  asm("mad.lo.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(y), "r"(z));
  return r;
}
__device__ __forceinline__ uint32_t hfma2(uint32_t x, uint32_t y, uint32_t z) {
  uint32_t r;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(y), "r"(z));
  return r;
}
__device__ __forceinline__ uint32_t hmul2(uint32_t x, uint32_t y) {
  uint32_t r;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(y));
  return r;
}
// |a| as in the plain kernel's ||A||_inf estimate (ir.cu): fp32 from the top word
__device__ __forceinline__ float abs_est(int hi) {
  const int t = (hi & 0x7fffffff) - (896 << 20);
  return t > 0 ? __int_as_float(min(t, 0x7f7fffff >> 3) << 3) : 0.0f;
}

struct GemvTc {
  int64_t n;
  const double* X; int64_t ldx;
  const uint8_t* dig;
  const int* ex;
  const int* fr;
  double* P;          // [piece][rhs][n]
  float* RS;          // [piece][n] estimated |A| row sums (kAbs)
  GemvSplit split;
  // the constants 1, -1 and 2048 as run-time values: multiply-adds by them run
  // on the FMA pipe, while adds and shifts would share the integer pipe that
  // bounds this kernel
  int one, minus;
  uint32_t k2048;
  uint32_t* status;
  long long wait_polls;
  unsigned long long wait_ns;
  Gate gate;
};

template <int K, bool kAbs>
__global__ void __launch_bounds__(kThr, 1) gemv_tc_kernel(const __grid_constant__ CUtensorMap tmA, GemvTc p) {
  if (p.gate.flag) {
    pdl_wait();
    if (p.gate.closed()) return;
  }
  extern __shared__ uint8_t raw_smem[];
  uint8_t* smem = raw_smem + ((1024u - (smem_u32(raw_smem) & 1023u)) & 1023u);
  uint8_t* ring = smem + kBArea;                                                    // [group][stage][8 columns][128 rows]
  long long* hl = reinterpret_cast<long long*>(ring + kGroups * kStages * kStage);  // [2][K][512]
  int* exps = reinterpret_cast<int*>(hl + 2 * K * kTileRows);                       // [buffer][kExpW]
  uint64_t* bars = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(exps) + kBBufs * kExp);
  uint32_t* slot = reinterpret_cast<uint32_t*>(bars + kBars);
  volatile uint32_t* dead = slot + 1;   // a wait ran out: no further waits (the results are void, the call reports it)
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = warp >> 2, tg = tid & (kRowsT - 1);
  // A group's MMAs and its loads are issued by one thread each, in another warp in each group: warps 0 of
  // all groups share a scheduler, and with their MMAs all issued there the product took 8 % longer
  const int mma_thread = 32 * g, load_thread = 32 * ((g + 2) & 3);
  const uint32_t bar0 = smem_u32(bars);
  auto b_full = [&](int b) { return bar0 + 8u * (uint32_t)b; };
  auto b_empty = [&](int b) { return bar0 + 8u * (uint32_t)(kBBufs + b); };
  auto a_full = [&](int gg, int s) { return bar0 + 8u * (uint32_t)(2 * kBBufs + gg * kStages + s); };
  const uint32_t bar_mma = bar0 + 8u * (uint32_t)(2 * kBBufs + kGroups * kStages + g);
  const uint32_t bar_drain = bar_mma + 8u * (uint32_t)kGroups;
  auto digits_at = [&](int b) { return smem_u32(smem) + (uint32_t)(1 + b * (kSlices + 1)) * 1024; };

  for (int i = tid * 16; i < kBArea; i += kThr * 16) *reinterpret_cast<uint4*>(smem + i) = make_uint4(0, 0, 0, 0);
  if (tid == 0) {
    *dead = 0;
    for (int b = 0; b < kBBufs; ++b) { mbar_init(b_full(b), 1); mbar_init(b_empty(b), kGroups); }
    for (int k = 0; k < kGroups; ++k) {
      for (int s = 0; s < kStages; ++s) mbar_init(a_full(k, s), 1);
      mbar_init(bar0 + 8u * (uint32_t)(2 * kBBufs + kGroups * kStages + k), 1);
      mbar_init(bar0 + 8u * (uint32_t)(2 * kBBufs + kGroups * kStages + kGroups + k), 1);
    }
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  fence_async_smem();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  pdl_wait();
  pdl_trigger();

  // true when the phase completed; false (and the dead flag) when the wait ran out
  auto wait = [&](uint32_t bar, uint32_t parity) {
    if (mbar_try(bar, parity)) return true;
    if (*dead) return false;
    if (mbar_wait(bar, parity, p.wait_polls, p.wait_ns)) return true;
    *dead = 1;
    atomicOr(p.status, kErrTimeout);
    return false;
  };
  // hardly a column of X alike for the right-hand sides: fp64 FMAs throughout
  const bool plain = K > 1 && 8ll * p.fr[8] > 7 * p.n;
  const int nkb = p.split.blocks;
  // a range's blocks w0 .. wend - 1 of the row tiles' concatenated lists, and how many stages and
  // digit buffers were used before it
  int w0 = 0, wend = 0;
  uint32_t a0 = 0, b0 = 0;
  {
    const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;
    const uint32_t ta = tmem + kTmA * g, td = tmem + kTmD + 64 * g;
    uint32_t apos = 0, bpos = 0, issued = 0;   // stages and digit buffers used, commits
    uint32_t a_loads = 0, b_loads = 0;         // next uses to load (load_thread)
    uint32_t fills_a[kStages] = {}, fills_b[kBBufs] = {};   // loads issued into each
    // A is read once: its lines leave L2 first, and the factors and inverses that the
    // preconditioner reads next stay
    uint64_t stream_policy;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(stream_policy));
    auto count_fill = [](auto& f, int k) {
#pragma unroll
      for (int i = 0; i < (int)(sizeof(f) / sizeof(f[0])); ++i) f[i] += i == k;
    };
    // columns of stage use q (of load_thread) and digits of block use q (of group 0's)
    auto load_a = [&](uint32_t q) {
      const int lw = w0 + (int)((q - a0) / (kBlk / kCols));
      if (lw >= wend || *dead) return;
      const int tile = lw / nkb, kb = lw - tile * nkb, s = q % kStages;
      count_fill(fills_a, s);
      mbar_expect_tx(a_full(g, s), kStage);
      tma_load_2d_stream(smem_u32(ring) + (g * kStages + s) * kStage, &tmA, tile * kTileRows + g * kRowsT,
                         kb * kBlk + (int)((q - a0) % (kBlk / kCols)) * kCols, a_full(g, s), stream_policy);
    };
    auto load_b = [&](uint32_t q) {
      const int lw = w0 + (int)(q - b0);
      if (lw >= wend || *dead) return;
      const int kb = lw % nkb, b = q % kBBufs;
      if (q >= kBBufs && !wait(b_empty(b), (q / kBBufs - 1) & 1)) return;
      count_fill(fills_b, b);
      mbar_expect_tx(b_full(b), kDig + kExp);
      bulk_load(digits_at(b), p.dig + (size_t)kb * kDig, kDig, b_full(b));
      bulk_load(smem_u32(exps) + b * kExp, reinterpret_cast<const uint8_t*>(p.ex) + (size_t)kb * kExp, kExp, b_full(b));
    };
    auto wait_mma = [&]() {
      if (issued) wait(bar_mma, (issued - 1) & 1);
      tc_fence_after();
    };
    // (a grid below the number of ranges, with an SM budget, takes several in turn: the sums do
    // not depend on the grid)
    for (int range = blockIdx.x; range < p.split.ctas; range += gridDim.x) {
    int w = w0 = p.split.begin(range);
    wend = p.split.begin(range + 1);
    a0 = apos;
    b0 = bpos;
    if (tg == load_thread) {
      for (a_loads = a0; a_loads < a0 + kStages; ++a_loads) load_a(a_loads);
      if (g == 0 && !plain)
        for (b_loads = b0; b_loads < b0 + kBBufs - 1; ++b_loads) load_b(b_loads);
    }
    while (w < wend) {
      int tile = w / nkb, kb0 = w - tile * nkb;
      const int kb1 = min(nkb, kb0 + wend - w);
      w += kb1 - kb0;
      const int piece = range - p.split.first_cta(tile);
      const int64_t row = (int64_t)tile * kTileRows + tid;
      double facc[K];                 // products taken in fp64, and the folded integers
#pragma unroll
      for (int r = 0; r < K; ++r) {
        facc[r] = 0.0;
        hl[r * kTileRows + tid] = 0;
        hl[(K + r) * kTileRows + tid] = 0;
      }
      float rowsum = 0.0f;
      int E = 0, over = 0, otop = 0;  // running exponent; entries above it so far and their largest
      bool pend = false, pend_bad = false;   // a block's D is not taken yet / is not to be used
      int pend_E = 0;                        // its E
      // integers so far into fp64: 2^(E - 1037 + f_r) (H 2^-24 + L 2^-56)
      auto fold = [&]() {
#pragma unroll
        for (int r = 0; r < K; ++r) {
          const long long H = hl[r * kTileRows + tid], L = hl[(K + r) * kTileRows + tid];
          if ((H | L) != 0) facc[r] += scalbn(__fma_rn((double)H, 0x1p-24, (double)L * 0x1p-56), E - 1037 + p.fr[r]);
          hl[r * kTileRows + tid] = 0;
          hl[(K + r) * kTileRows + tid] = 0;
        }
      };
      // a stage's columns, from j on, in fp64, for the rows that want it (`mine`).  all: zero entries
      // count (x may be non-finite).  A row without an E keeps its two largest scaled exponents among
      // the robust columns in otop, over
      auto fp64_stage = [&](const double* col, const int* ej, int64_t j, bool all, bool mine) {
        if (!all) {
          uint32_t any = 0;
#pragma unroll
          for (int c = 0; c < kCols; ++c)
            any |= ((uint32_t)__double2hiint(col[c * kRowsT]) << 1) | (uint32_t)__double2loint(col[c * kRowsT]);
          if (any == 0) return;
        }
        const int cols = mine ? (int)min((int64_t)kCols, p.n - j) : 0;
#pragma unroll 1
        for (int c = 0; c < cols; ++c) {
          const double a = col[c * kRowsT];
#pragma unroll
          for (int r = 0; r < K; ++r) facc[r] = __fma_rn(a, __ldg(p.X + j + c + r * p.ldx), facc[r]);
          if (plain) {
            if (kAbs) rowsum += abs_est(__double2hiint(a));
          } else if (E < kMinE) {
            const int t = (__double2hiint(a) & 0x7fffffff) + ej[kBlk + c];
            over = max(over, min(otop, t));
            otop = max(otop, t);
          }
        }
      };
      auto flush = [&]() {   // the pending block's D, complete, into H and L
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t d[4][8];
#pragma unroll
          for (int v = 0; v < 4; ++v) tmem_ld8(td + lane_off + 8 * (4 * h + v), d[v]);
          // the registers pass through the wait: nothing reads them before it
          asm volatile("tcgen05.wait::ld.sync.aligned;"
                       : "+r"(d[0][0]), "+r"(d[0][1]), "+r"(d[0][2]), "+r"(d[0][3]), "+r"(d[0][4]), "+r"(d[0][5]),
                         "+r"(d[0][6]), "+r"(d[0][7]), "+r"(d[1][0]), "+r"(d[1][1]), "+r"(d[1][2]), "+r"(d[1][3]),
                         "+r"(d[1][4]), "+r"(d[1][5]), "+r"(d[1][6]), "+r"(d[1][7]), "+r"(d[2][0]), "+r"(d[2][1]),
                         "+r"(d[2][2]), "+r"(d[2][3]), "+r"(d[2][4]), "+r"(d[2][5]), "+r"(d[2][6]), "+r"(d[2][7]),
                         "+r"(d[3][0]), "+r"(d[3][1]), "+r"(d[3][2]), "+r"(d[3][3]), "+r"(d[3][4]), "+r"(d[3][5]),
                         "+r"(d[3][6]), "+r"(d[3][7])
                       :
                       : "memory");
          if (!pend_bad) {
#pragma unroll
            for (int r = 0; r < K; ++r) {
              int v[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) v[k] = __float2int_rn(__uint_as_float(d[k][r]));
              const long long sum =
                  (long long)v[0] * (1 << 24) + (long long)v[1] * (1 << 16) + (long long)v[2] * 256 + v[3];
              if (pend_E == E) hl[(h * K + r) * kTileRows + tid] += sum;
              else facc[r] += scalbn((double)sum, pend_E - 1037 - (h ? 56 : 24) + p.fr[r]);
            }
          }
        }
        pend = false;
      };

      if (plain) {
        for (int q = 4 * kb0; q < 4 * kb1; ++q, ++apos) {
          const uint32_t st = apos % kStages;
          wait(a_full(g, st), (apos / kStages) & 1);
          fp64_stage(reinterpret_cast<const double*>(ring + (g * kStages + st) * kStage) + tg, exps, (int64_t)q * kCols, true,
                     true);
          group_barrier(g);
          if (tg == load_thread) load_a(a_loads++);
        }
        kb0 = kb1;
      }
      for (int kb = kb0; kb < kb1; ++kb, ++bpos) {
        const int bb = bpos % kBBufs;
        wait(b_full(bb), (bpos / kBBufs) & 1);
        const int* e0 = exps + bb * kExpW;
        if (kb == kb0) {
          // E from the first 16 columns: one above the largest of the robust ones, unless that
          // one stands alone (a dominant diagonal)
          wait(a_full(g, apos % kStages), (apos / kStages) & 1);
          const double* col = reinterpret_cast<const double*>(ring + (g * kStages + apos % kStages) * kStage) + tg;
          int m1 = INT_MIN, m2 = INT_MIN;
#pragma unroll
          for (int c = 0; c < kCols; ++c) {
            const int t = (__double2hiint(col[c * kRowsT]) & 0x7fffffff) + e0[kBlk + c];
            m2 = max(m2, min(m1, t));
            m1 = max(m1, t);
          }
          m1 >>= 20;
          m2 >>= 20;
          E = min(m1 - m2 <= 3 ? m1 + 1 : m2 + 2, kMaxE + 1);
        }
        const bool odd_x = e0[2 * kBlk] != 0;
        const bool bad = odd_x || E < kMinE || E > kMaxE;   // this block in fp64
        const int etop = E * (1 << 20) + 0xfffff;
        if (E < kMinE) over = otop = INT_MIN;
        // one branch per warp and behind the digits: a row's own ahead of them cost every block 4 %
        const bool any_bad = __any_sync(0xffffffffu, bad);
#pragma unroll 1
        for (int sub = 0; sub < 4; ++sub, ++apos) {
          const uint32_t st = apos % kStages;
          wait(a_full(g, st), (apos / kStages) & 1);
#pragma unroll
          for (int half = 0; half < 2; ++half) {   // 8 columns at a time: their digits are 32 registers
            const double* col = reinterpret_cast<const double*>(ring + (g * kStages + st) * kStage) + 8 * half * kRowsT + tg;
            const int* ej = e0 + 16 * sub + 8 * half;
            int tmax = INT_MIN;
            uint32_t sl[kSlices][4];
#pragma unroll
            for (int c4 = 0; c4 < 2; ++c4) {
              const int4 ec4 = *reinterpret_cast<const int4*>(ej + 4 * c4);
              const int ec[4] = {ec4.x, ec4.y, ec4.z, ec4.w};
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                uint32_t vh[2], vl[2], hi2[2];
                int t2[2];
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                  const double a = col[(4 * c4 + 2 * h + b) * kRowsT];
                  const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
                  hi2[b] = hi;
                  if (kAbs) rowsum += abs_est((int)hi);
                  t2[b] = mad((int)(hi & 0x7fffffffu), p.one, ec[2 * h + b]);
                  // significand with its leading one at bit 63, then down to 2^E's scale; a zero or
                  // subnormal entry shifts out (E >= kMinE), and so does one above 2^E (a negative
                  // count, read unsigned)
                  const uint64_t ml = (uint64_t)lo * p.k2048;
                  const uint64_t m =
                      ((uint64_t)((hi | 0x00100000u) * p.k2048 + (uint32_t)(ml >> 32)) << 32) | (uint32_t)ml;
                  uint64_t v;
                  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"((uint32_t)(mad(t2[b], p.minus, etop) >> 20)));
                  vh[b] = (uint32_t)(v >> 32);
                  vl[b] = (uint32_t)v;
                }
                tmax = __vimax3_s32(tmax, t2[0], t2[1]);
                // digits as fp16: 0x6400 | u is 1024 + u; times the sign, minus 1024 times the sign
                const uint32_t sg = __byte_perm(hi2[0], hi2[1], 0x7030);
                const uint32_t one = (sg & 0x80008000u) | 0x3c003c00u, off = hmul2(one, 0xe400e400u);
#pragma unroll
                for (int s = 0; s < kSlices; s += 2) {   // two bytes of both entries, then each with the exponent byte
                  const uint32_t by = s < 4 ? __byte_perm(vh[0], vh[1], s == 0 ? 0x6723 : 0x4501)
                                            : __byte_perm(vl[0], vl[1], s == 4 ? 0x6723 : 0x4501);
                  const uint32_t u0 = __byte_perm(by, 0x64646464u, 0x4240), u1 = __byte_perm(by, 0x64646464u, 0x4341);
                  sl[s][2 * c4 + h] = hfma2(u0, one, off);
                  sl[s + 1][2 * c4 + h] = hfma2(u1, one, off);
                }
              }
            }
            if (tmax > etop && !bad) {   // entries above 2^E: their products in fp64
              // every lane its own columns, so that a warp on the diagonal takes one round
              uint32_t above = 0;
#pragma unroll
              for (int c = 0; c < 8; ++c)
                above |= (uint32_t)((__double2hiint(col[c * kRowsT]) & 0x7fffffff) + ej[c] > etop) << c;
              // columns past the last one are zeros, but after a wait that ran out the stage and the
              // exponents hold anything: x has n entries
              const int64_t left = p.n - ((int64_t)kb * kBlk + 16 * sub + 8 * half);
              if (left < 8) above &= left > 0 ? (1u << left) - 1u : 0u;
              while (above) {
                const int c = __ffs((int)above) - 1;
                above &= above - 1;
                const double a = col[c * kRowsT];
                const double* x = p.X + (int64_t)kb * kBlk + 16 * sub + 8 * half + c;
#pragma unroll
                for (int r = 0; r < K; ++r) facc[r] = __fma_rn(a, __ldg(x + r * p.ldx), facc[r]);
                if (ej[kBlk + c] == ej[c]) {
                  ++over;
                  otop = max(otop, (__double2hiint(a) & 0x7fffffff) + ej[c]);
                }
              }
            }
            if (half == 0) {
              wait_mma();                    // the digits' TMEM is free, and D complete
              if (sub == 0 && pend) flush();
            }
#pragma unroll
            for (int s = 0; s < kSlices; ++s) tmem_st4(ta + lane_off + 8 * s + 4 * half, sl[s]);
          }
          if (any_bad)
            fp64_stage(reinterpret_cast<const double*>(ring + (g * kStages + st) * kStage) + tg, e0 + kCols * sub,
                       (int64_t)kb * kBlk + kCols * sub, odd_x, bad);
          asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
          tc_fence_before();
          group_barrier(g);
          if (tg == mma_thread) {
            tc_fence_after();
            const uint32_t bd = digits_at(bb) + 32 * sub;
#pragma unroll
            for (int s = 0; s < kSlices; ++s)
              // D's columns from 8 s on (an odd s starts a zero group and 8 columns earlier, so
              // that the column counts are multiples of 16)
              tc_mma_ts(td + 16 * (s / 2), ta + 8 * s, sdesc_sw128(bd - (s & 1) * 1024),
                        make_idesc(0, 64 - 16 * (s / 2)), sub > 0 || s > 0);
            if (sub == 3) tc_commit(b_empty(bb));
            tc_commit(bar_mma);   // the last one, which the drain below waits for
          } else if (tg == load_thread) {   // every thread of the group has read this stage
            load_a(a_loads++);
            if (g == 0 && sub == 2) load_b(b_loads++);
          }
          ++issued;
        }
        pend = true;
        pend_bad = bad;
        pend_E = E;
        if (E < kMinE) {   // nothing in H, L or D yet
          E = max(E, min((over >> 20) + 1, kMaxE + 1));
          over = otop = 0;
        } else if (over >= 3) {
          fold();
          E = min(otop >> 20, kMaxE + 1);
          over = otop = 0;
        }
      }
      if (pend) {
        wait_mma();
        flush();
        tc_fence_before();
      }
      fold();
      if (row < p.n) {
#pragma unroll
        for (int r = 0; r < K; ++r) p.P[((int64_t)piece * K + r) * p.n + row] = facc[r];
        if (kAbs) p.RS[(int64_t)piece * p.n + row] = rowsum;
      }
    }
    }
    // every MMA issued has completed before tensor memory is freed, and every copy has
    // landed before the CTA exits (default bound)
    if (issued && !mbar_wait(bar_mma, (issued - 1) & 1)) atomicOr(p.status, kErrTimeout);
    // Where a wait ran out, several commits can be open, and bar_mma's parity is that of the one before
    // the last as well: the issuing thread commits once more, to a barrier used for nothing else.  (If it
    // does not see the flag, each of its own waits ended before its next MMAs, and one commit at most was open.)
    if (tg == mma_thread && issued && *dead) {
      tc_commit(bar_drain);
      if (!mbar_wait(bar_drain, 0)) atomicOr(p.status, kErrTimeout);
    }
    if (tg == load_thread && *dead) {
      for (int s = 0; s < kStages; ++s)
        if (fills_a[s] && !mbar_wait(a_full(g, s), (fills_a[s] - 1) & 1)) atomicOr(p.status, kErrTimeout);
      for (int b = 0; b < kBBufs; ++b)
        if (fills_b[b] && !mbar_wait(b_full(b), (fills_b[b] - 1) & 1)) atomicOr(p.status, kErrTimeout);
    }
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

int sm_count() {
  static std::atomic<int> sms{0};
  int v = sms.load();
  if (!v) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    sms.store(v);
  }
  return v;
}

template <int K, bool kAbs>
cudaError_t launch_k(const CUtensorMap& tm, const GemvTc& p, cudaStream_t st, bool pdl) {
  // one value for every call: concurrent solves on other threads set the same
  cudaError_t e = cudaFuncSetAttribute(gemv_tc_kernel<K, kAbs>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)gemv_smem<K>());
  if (e != cudaSuccess) return e;
  const int budget = sm_budget();
  const int grid = budget > 0 ? std::min(budget, p.split.ctas) : p.split.ctas;
  return launch_vec(pdl, gemv_tc_kernel<K, kAbs>, dim3(grid), dim3(kThr), gemv_smem<K>(), st, tm, p);
}

}  // namespace

size_t gemv_tc_bytes(int64_t n) { return (size_t)cdiv<int64_t>(n, kBlk) * (kDig + kExp) + 64; }

bool gemv_tc_split(int64_t n, const double* A, int64_t lda, int max_pieces, GemvSplit* split) {
  // TMA: 16-byte aligned columns
  if (((uintptr_t)A & 15) || (lda & 1)) return false;
  const int tiles = (int)cdiv<int64_t>(n, kTileRows);
  split->blocks = (int)cdiv<int64_t>(n, kBlk);
  split->total = tiles * split->blocks;
  split->ctas = std::min(split->total, sm_count());
  // a tile meets at most this many CTAs' ranges
  return most_of(*split) <= max_pieces;
}

cudaError_t gemv_tc(int64_t n, int K, const double* A, int64_t lda, const double* X, int64_t ldx, bool abs_sums,
                    void* prep, double* P, void* RS, const GemvSplit& split, uint32_t* status, cudaStream_t st, bool pdl, Gate gate,
                    Gate live) {
  const int nkb = (int)cdiv<int64_t>(n, kBlk);
  GemvTc p{};
  p.n = n; p.X = X; p.ldx = ldx;
  uint8_t* dig = (uint8_t*)prep;
  int* ex = (int*)(dig + (size_t)nkb * kDig);
  int* fr = ex + (size_t)nkb * kExpW;
  p.dig = dig; p.ex = ex; p.fr = fr;
  p.P = P; p.RS = (float*)RS;
  p.split = split;
  p.one = 1; p.minus = -1; p.k2048 = 2048;
  p.status = status;
  const WaitBudget wb = wait_budget();
  p.wait_polls = wb.polls;
  p.wait_ns = wb.ns;
  p.gate = gate;
  CUtensorMap tm;
  if (!encode_f64_map(&tm, A, n, n, lda, kRowsT, kCols)) return cudaErrorInvalidValue;
  count_launches(3);
  cudaError_t e = launch_vec(pdl, xscale_kernel, dim3(K), dim3(1024), 0, st, n, X, ldx, fr, gate, live);
  if (e == cudaSuccess) e = launch_vec(pdl, digit_kernel, dim3(nkb), dim3(512), 0, st, n, K, X, ldx, fr, dig, ex, gate);
  if (e != cudaSuccess) return e;
#define HPMXP_GEMV_K(KK) \
  case KK: return abs_sums ? launch_k<KK, true>(tm, p, st, pdl) : launch_k<KK, false>(tm, p, st, pdl)
  switch (K) {
    HPMXP_GEMV_K(1);
    HPMXP_GEMV_K(2);
    HPMXP_GEMV_K(3);
    HPMXP_GEMV_K(4);
    HPMXP_GEMV_K(5);
    HPMXP_GEMV_K(6);
    HPMXP_GEMV_K(7);
    HPMXP_GEMV_K(8);
    default: return cudaErrorInvalidValue;
  }
#undef HPMXP_GEMV_K
}

}  // namespace hpmxp
