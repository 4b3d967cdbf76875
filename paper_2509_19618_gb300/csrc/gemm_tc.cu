// Tensor-core product engine for the LU's panel and Schur-update products
// (section "Algorithmic Framework", Fig. 1: low-precision operands, fp32
// accumulation).  sm_103a: operands are staged into shared memory by TMA
// (128-byte swizzle, K-major), multiplied by tcgen05.mma issued from one
// thread with fp32 accumulators in tensor memory, and read back with
// tcgen05.ld by four epilogue warps.
//
// Persistent kernel, one CTA per SM, TI x 128 output tiles (TI = 128, or 256
// for the large 16-bit products) in a static round-robin order.  The MMA
// computes the TRANSPOSED tile (TMEM lane = output column j, TMEM column =
// output row i) so each epilogue thread owns consecutive rows of one column of
// the column-major output: the C tile is moved by TMA between HBM and
// 128-byte-swizzled shared boxes of 64 rows and the epilogue touches them with
// 16-byte, bank-conflict-free accesses.
//
// Large products of depth 512 run on pairs of CTAs (kPair): rank 0 issues the
// MMAs of both and commits to both CTAs' barriers; each CTA has its own producer,
// epilogue and C movers.  Both producers' loads complete on rank 0's barrier, so
// that the bytes of rank 1's shared memory are ordered before the MMAs that read
// them as those of its own are (no relay by a thread of rank 1, whose cluster-scope
// fences took 0.5 us a stage); rank 1's epilogue frees an accumulator, once per
// tile, by an arrival at cluster scope.
//
// Roles: warp 0 TMA producer of the operand ring; warp 1 TMEM owner and MMA
// issuer; warps 2..9 epilogue in two groups of four (warp w reads TMEM lanes
// 32*(w%4)..+31; group g takes rows TI/2 g .. of the tile); warps 10 and 11
// move the groups' C: loads ahead, stores behind, by 64-row segments (where C has
// one buffer; with three each group's first thread does).
// Accumulators are double buffered in TMEM (single buffered for 4-slice FP8),
// so the epilogue of one tile overlaps the MMAs of the next.  The E4M3
// variant keeps one accumulator per 128-deep K slice and folds them with the
// per-tile scales in the epilogue.
//
// Every wait is bounded (a poll count and a global-timer limit passed in
// TcParams); a wait that runs out sets kErrTimeout in the status word, skips
// the remaining work and still drains its copies and tensor-core work (with
// the default bound) and frees tensor memory before the CTA exits.
#include "tcgen05.h"

#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <mutex>

namespace hpmxp {
namespace {

constexpr int kTJ = 128;                      // output columns per tile (MMA M, TMEM lanes)
constexpr int kRowBytes = 128;                // K bytes per operand row per stage (one swizzle atom)
constexpr int kStageA = kTJ * kRowBytes;      // MMA A operand: rows j (16 KiB)
constexpr int kCBox = kTJ * 128;              // one C box: 128 bytes of rows x 128 columns (16 KiB)
constexpr int kEpiGroups = 2;                 // epilogue groups, one per half of the tile's rows
constexpr int kEpiThreads = 128;              // threads per epilogue group (one warp per TMEM lane quarter)
constexpr int kEpiWarps = kEpiThreads / 32;

// Tile height TI (output rows i per tile = MMA N): 128, or 256 for the large
// 16-bit products, where every operand byte an SM receives feeds twice the
// flops (the SM's operand intake is what bounds this kernel at K >= 256).
// CB: bytes per C element, 2 (the 16-bit factor storage) or 4 (an fp32
// trailing matrix: C = fl32(C - acc), 128-row tiles only).
// kPair: a cluster of two CTAs makes a tile of 256 rows and 256 columns, each
// its own 128 columns of the accumulator; each stages 128 of the rows i, so that
// an SM receives 32 instead of 48 KB per 64 of depth (953 -> 1182 TFLOP/s at
// order 28672, depth 512; the n = 32768 factorization 36.7 -> 32.1 ms).
template <int TI, int CB = 2, bool kPair = false>
struct TileCfg {
  static constexpr int kStages = kPair ? 5 : TI == 128 ? 4 : 3;
  static constexpr int kRowsB = kPair ? TI / 2 : TI;        // MMA B operand: rows i in this CTA
  static constexpr int kStageB = kRowsB * kRowBytes;        // (16 or 32 KiB)
  static constexpr int kBoxRows = 128 / CB;                 // rows of one 128-byte C box: 64 or 32
  static constexpr int kBoxes = TI / 2 / kBoxRows;          // C boxes per epilogue group
  static constexpr int kCTile = kEpiGroups * kBoxes * kCBox;  // 32, 64 KiB (16-bit) or 64 KiB (fp32)
  // C tile buffers; the 256-row and the fp32 tiles have room for one only
  static constexpr int kCBufs = (TI == 128 && CB == 2) ? 3 : 1;
  // who moves a group's C: a warp of its own, or with three buffers the group's first thread
  static constexpr bool kMover = kCBufs == 1;
  static constexpr int kThreads = 64 + kEpiGroups * (kEpiThreads + (kMover ? 32 : 0));
  static constexpr int kSegs = TI / 128;                    // 64-row segments of an epilogue group's TI/2 rows
  static constexpr int kSegBoxes = kBoxes / kSegs;          // C boxes of a segment
  static constexpr int kCSlots = kCBufs * kEpiGroups * kSegs;
  static constexpr int kBars = 2 * kStages + 5 + 2 * kCSlots;
  static constexpr size_t kSmem = 1024 + (size_t)kStages * (kStageA + kStageB) + (size_t)kCBufs * kCTile +
                                  8 * kBars + 16;
};
// 227 KB of dynamic shared memory per CTA; two TI-column fp32 accumulators in
// the 512 TMEM columns; a TMA box is at most 256 rows
static_assert(TileCfg<128>::kSmem <= 232448 && TileCfg<256>::kSmem <= 232448 && TileCfg<256, 2, true>::kSmem <= 232448 && TileCfg<128, 4>::kSmem <= 232448,
              "shared memory per CTA");
template <int TI>
constexpr bool tile_fits() { return 2 * TI <= 512 && TI <= 256 && TI % 128 == 0; }
static_assert(tile_fits<128>() && tile_fits<256>(), "two accumulators in TMEM, one TMA box per stage");

// Barrier of an epilogue group; true for all of its threads when v is true for all.
__device__ inline bool epi_all(int group, bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(1 + group), "n"(kEpiThreads)
      : "memory");
  return r != 0;
}

// 64 consecutive fp32 columns: two x32 loads in flight, one wait.
__device__ inline void tmem_ld64(uint32_t taddr, uint32_t (&r)[64]) {
#define HPMXP_LD32(OFF, B)                                                                                       \
  asm volatile(                                                                                                \
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, " \
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"            \
      : "=r"(r[B + 0]), "=r"(r[B + 1]), "=r"(r[B + 2]), "=r"(r[B + 3]), "=r"(r[B + 4]), "=r"(r[B + 5]),         \
        "=r"(r[B + 6]), "=r"(r[B + 7]), "=r"(r[B + 8]), "=r"(r[B + 9]), "=r"(r[B + 10]), "=r"(r[B + 11]),       \
        "=r"(r[B + 12]), "=r"(r[B + 13]), "=r"(r[B + 14]), "=r"(r[B + 15]), "=r"(r[B + 16]), "=r"(r[B + 17]),   \
        "=r"(r[B + 18]), "=r"(r[B + 19]), "=r"(r[B + 20]), "=r"(r[B + 21]), "=r"(r[B + 22]), "=r"(r[B + 23]),   \
        "=r"(r[B + 24]), "=r"(r[B + 25]), "=r"(r[B + 26]), "=r"(r[B + 27]), "=r"(r[B + 28]), "=r"(r[B + 29]),   \
        "=r"(r[B + 30]), "=r"(r[B + 31])                                                                        \
      : "r"(taddr + OFF))
  HPMXP_LD32(0u, 0);
  HPMXP_LD32(32u, 32);
#undef HPMXP_LD32
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                 "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                 "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                 "+r"(r[29]), "+r"(r[30]), "+r"(r[31]), "+r"(r[32]), "+r"(r[33]), "+r"(r[34]), "+r"(r[35]),
                 "+r"(r[36]), "+r"(r[37]), "+r"(r[38]), "+r"(r[39]), "+r"(r[40]), "+r"(r[41]), "+r"(r[42]),
                 "+r"(r[43]), "+r"(r[44]), "+r"(r[45]), "+r"(r[46]), "+r"(r[47]), "+r"(r[48]), "+r"(r[49]),
                 "+r"(r[50]), "+r"(r[51]), "+r"(r[52]), "+r"(r[53]), "+r"(r[54]), "+r"(r[55]), "+r"(r[56]),
                 "+r"(r[57]), "+r"(r[58]), "+r"(r[59]), "+r"(r[60]), "+r"(r[61]), "+r"(r[62]), "+r"(r[63])
               :
               : "memory");
}

struct TcParams {
  int M, N, nkb;          // output rows, columns, K stages (128 bytes of K each)
  int tiles_i, ntiles;
  int split;              // tiles from here on belong to the launch's second product (TcSecond)
  int mode;
  float sign;
  int fmt;
  int fp8;                // E4M3 operands: one accumulator per stage (= 128-deep slice)
  int nbuf;               // TMEM accumulator buffers (1 or 2)
  uint32_t acc_cols;      // TMEM columns per accumulator buffer
  uint32_t ncols;         // TMEM columns allocated
  int has_c;              // write (and for kEpiSub read) the column-major C through tmC
  uint16_t* R; int64_t ldr;
  const float* sA; int sa_ld;
  const float* sB; int sb_ld;
  uint32_t* status;
  long long wait_polls;            // bound of the pipeline waits (the drain waits keep the defaults)
  unsigned long long wait_ns;
  // measurement: [0] the earliest CTA start after the stream dependency, [1]
  // all-ones minus the latest CTA end (global timer, ns; both kept by
  // atomicMin from all-ones), NULL when not measured
  unsigned long long* span;
};

// The second of two independent products of one launch (same depth, mode and
// types): the row panel and the column panel of a step, 128 wide each, would
// otherwise take turns, 7 us for a second launch of a few tiles.
struct TcSecond {
  CUtensorMap a, b, c;
  int M, N, tiles_i;
  uint16_t* R; int64_t ldr;
};

// Two floats rounded to nearest even into one 32-bit word of 16-bit values (lo
// in the low half): one packed conversion instruction.
__device__ inline uint32_t pack16x2(float lo, float hi, int fmt) {
  uint32_t r;
  if (fmt == kBF16) asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  else asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// Where tile t of the launch is: its product's tensor maps, its output origin
// and that product's bounds (one product, or the items of a grouped launch).
struct TileLoc {
  const CUtensorMap* a;
  const CUtensorMap* b;
  const CUtensorMap* c;
  int i0, j0, M, N;
  uint16_t* R;
  int64_t ldr;
};

template <int TI, int CB, bool kPair>
__global__ void __launch_bounds__(TileCfg<TI, CB, kPair>::kThreads, 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmC, TcParams p, const GemmGroupItem* __restrict__ items,
               int nitems, const __grid_constant__ TcSecond second) {
  using Cfg = TileCfg<TI, CB, kPair>;
  constexpr int kStages = Cfg::kStages, kStageB = Cfg::kStageB, kCTile = Cfg::kCTile, kCBufs = Cfg::kCBufs;
  constexpr int kBoxes = Cfg::kBoxes, kBoxRows = Cfg::kBoxRows, kSegs = Cfg::kSegs, kSegBoxes = Cfg::kSegBoxes;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + ((1024u - (raw & 1023u)) & 1023u);   // swizzle atoms need 1024-byte alignment
  const uint32_t sOpA = smem_u32(smem);                            // [kStages][rows j][128 B]
  const uint32_t sOpB = sOpA + kStages * kStageA;                  // [kStages][rows i][128 B]
  const uint32_t sC = sOpB + kStages * kStageB;                    // [kCBufs][group][box][cols j][128 B]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * (kStageA + kStageB) + kCBufs * kCTile);
  const uint32_t bar0 = smem_u32(bars);
  auto full = [&](int s) { return bar0 + 8u * (uint32_t)s; };
  auto empty = [&](int s) { return bar0 + 8u * (uint32_t)(kStages + s); };
  auto acc_full = [&](int b) { return bar0 + 8u * (uint32_t)(2 * kStages + b); };
  auto acc_empty = [&](int b) { return bar0 + 8u * (uint32_t)(2 * kStages + 2 + b); };
  // segment h of group g in buffer b: its C is there (or the buffer is free, where C is not read);
  // the epilogue's four warps are done with it
  auto c_full = [&](int b, int g, int h) {
    return bar0 + 8u * (uint32_t)(2 * kStages + 4 + (b * kEpiGroups + g) * kSegs + h);
  };
  auto c_done = [&](int b, int g, int h) { return c_full(b, g, h) + 8u * (uint32_t)Cfg::kCSlots; };
  const uint32_t mma_drain = bar0 + 8u * (uint32_t)(2 * kStages + 4 + 2 * Cfg::kCSlots);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + Cfg::kBars);
  // (pair) stages loaded by the producers of ranks 0 and 1 and used by the MMAs, when they have ended
  volatile int* ended = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = kPair ? (int)cluster_rank() : 0;
  // tiles first(), first() + stride(), ...: read where used (as variables held from here on they
  // cost the small products of the chain 2 us each)
  auto first = [] { return kPair ? (int)blockIdx.x >> 1 : (int)blockIdx.x; };
  auto stride = [] { return kPair ? (int)gridDim.x >> 1 : (int)gridDim.x; };

  // tile t -> its product (grouped launch: the last item starting at or before t)
  auto locate = [&](int t) {
    TileLoc L;
    if (items == nullptr && t >= p.split) {
      t -= p.split;
      L.a = &second.a; L.b = &second.b; L.c = &second.c;
      L.i0 = (t % second.tiles_i) * TI; L.j0 = (t / second.tiles_i) * kTJ;
      L.M = second.M; L.N = second.N; L.R = second.R; L.ldr = second.ldr;
    } else if (items == nullptr) {
      L.a = &tmA; L.b = &tmB; L.c = &tmC;
      L.i0 = (t % p.tiles_i) * TI; L.j0 = ((t / p.tiles_i) * (kPair ? 2 : 1) + rank) * kTJ;
      L.M = p.M; L.N = p.N; L.R = p.R; L.ldr = p.ldr;
    } else {
      int lo = 0, hi = nitems - 1;
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (items[mid].tile_begin <= t) lo = mid; else hi = mid - 1;
      }
      const GemmGroupItem& g = items[lo];
      const int lt = t - g.tile_begin;
      L.a = reinterpret_cast<const CUtensorMap*>(g.maps[0]);
      L.b = reinterpret_cast<const CUtensorMap*>(g.maps[1]);
      L.c = reinterpret_cast<const CUtensorMap*>(g.maps[2]);
      L.i0 = (lt % g.tiles_i) * TI; L.j0 = (lt / g.tiles_i) * kTJ;
      L.M = g.M; L.N = g.N; L.R = (uint16_t*)g.R; L.ldr = g.ldr;
    }
    return L;
  };
  // the items' tensor maps were written to global memory before the launch:
  // acquire them for the tensor-map proxy before the first TMA through them
  auto acquire_maps = [&](int which) {
    for (int it = 0; items != nullptr && it < nitems; ++it)
      asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"((uint64_t)items[it].maps[which])
                   : "memory");
  };

  if (warp == 0 && lane == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full(s), 1); mbar_init(empty(s), 1); }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full(b), 1);
      mbar_init(acc_empty(b), (kPair ? 2 : 1) * kEpiGroups * kEpiWarps);
    }
    for (int b = 0; b < kCBufs; ++b)
      for (int g = 0; g < kEpiGroups; ++g)
        for (int h = 0; h < kSegs; ++h) {
          mbar_init(c_full(b, g, h), 1);
          mbar_init(c_done(b, g, h), kEpiWarps);
        }
    mbar_init(mma_drain, 1);
    fence_mbar_init();
    if (items == nullptr) {
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmA) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmB) : "memory");
      if (p.has_c) asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmC) : "memory");
    }
  }
  if (warp == 1) {
    if constexpr (kPair) {
      tmem_alloc_pair(smem_u32(tmem_slot), p.ncols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(tmem_slot), p.ncols);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (kPair) cluster_sync();   // both CTAs' barriers are initialised
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // the setup above may run while the previous kernel of the stream finishes;
  // no global memory is touched before it has completed
  pdl_wait();
  pdl_trigger();
  if (p.span && threadIdx.x == 0) atomicMin(p.span, global_ns());

  // operand ring: stage s holds K bytes [128 kb, +128) of the tile's rows j (A) and rows i (B);
  // pos: ring position over all tiles of this CTA
  auto load_stage = [&](const TileLoc& L, int kb, long long pos) {
    const int s = (int)(pos % kStages);
    if constexpr (kPair) {
      if (rank == 0) mbar_expect_tx(full(s), 2 * (kStageA + kStageB));
      const uint32_t bar = smem_at(full(s), 0);
      tma_load_2d_pair(sOpA + s * kStageA, L.b, kb * (kRowBytes / 2), L.j0, bar);
      tma_load_2d_pair(sOpB + s * kStageB, L.a, kb * (kRowBytes / 2), L.i0 + rank * Cfg::kRowsB, bar);
    } else {
      mbar_expect_tx(full(s), kStageA + kStageB);
      tma_load_2d(sOpA + s * kStageA, L.b, kb * (kRowBytes / 2), L.j0, full(s));
      tma_load_2d(sOpB + s * kStageB, L.a, kb * (kRowBytes / 2), L.i0, full(s));
    }
  };
  // the last load of every stage has landed before the CTA (or its pair) can exit
  auto drain_loads = [&](long long pos) {
    for (long long q = (pos > kStages ? pos - kStages : 0); q < pos; ++q)
      if (!mbar_wait(full((int)(q % kStages)), (uint32_t)((q / kStages) & 1))) atomicOr(p.status, kErrTimeout);
  };
  auto report_end = [&](int which, long long pos) {
    for (int r = 0; r < 2; ++r) store_at(smem_at(smem_u32(tmem_slot + 1 + which), (uint32_t)r), (int)pos);
  };

  // segment h of group g's C of a tile, in buffer b: its boxes, rows, load and store
  const bool load_c = p.has_c && p.mode == kEpiSub;
  auto c_box = [&](int b, int g, int h, int k) { return sC + b * kCTile + (g * kBoxes + h * kSegBoxes + k) * kCBox; };
  auto c_row = [&](int g, int h, int k) { return (TI / 2) * g + 64 * h + kBoxRows * k; };
  auto load_c_seg = [&](const TileLoc& L, int b, int g, int h) {
    mbar_expect_tx(c_full(b, g, h), kSegBoxes * kCBox);
#pragma unroll
    for (int k = 0; k < kSegBoxes; ++k)
      tma_load_2d(c_box(b, g, h, k), L.c, L.i0 + c_row(g, h, k), L.j0, c_full(b, g, h));
  };
  auto store_c_seg = [&](const TileLoc& L, int b, int g, int h) {
#pragma unroll
    for (int k = 0; k < kSegBoxes; ++k) tma_store_2d(L.c, L.i0 + c_row(g, h, k), L.j0, c_box(b, g, h, k));
  };

  if (warp == 0) {
    if (lane == 0) {
      long long pos = 0;
      bool ok = true;
      acquire_maps(0);
      acquire_maps(1);
      for (int t = first(); t < p.ntiles && ok; t += stride()) {
        const TileLoc L = locate(t);
        for (int kb = 0; kb < p.nkb; ++kb, ++pos) {
          const int s = (int)(pos % kStages);
          const long long use = pos / kStages;
          if (use > 0 && !mbar_wait(empty(s), (uint32_t)((use - 1) & 1), p.wait_polls, p.wait_ns)) {
            ok = false;
            break;
          }
          load_stage(L, kb, pos);
        }
      }
      if (!ok) atomicOr(p.status, kErrTimeout);
      if constexpr (kPair) report_end(rank, pos);   // drained below, together
      else drain_loads(pos);
    }
  } else if (kPair && warp == 1 && rank == 1) {
    // the MMAs are issued by rank 0
  } else if (warp == 1) {
    if (lane == 0) {
      auto commit = [](uint32_t bar) {
        if constexpr (kPair) tc_commit_pair(bar);
        else tc_commit(bar);
      };
      const uint32_t idesc = p.fp8 ? make_idesc(0, TI) : make_idesc(p.fmt == kBF16 ? 1u : 0u, TI, kPair ? 256 : 128);
      long long pos = 0;
      bool ok = true;
      int local = 0;
      for (int t = first(); t < p.ntiles && ok; t += stride(), ++local) {
        const int ab = local % p.nbuf, ause = local / p.nbuf;
        const uint32_t aph = (uint32_t)((ause - 1) & 1);
        if (ause > 0 &&
            !bounded_wait([&] { return kPair ? mbar_try_cluster(acc_empty(ab), aph) : mbar_try(acc_empty(ab), aph); },
                          p.wait_polls, p.wait_ns)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d0 = tmem + (uint32_t)ab * p.acc_cols;
        for (int kb = 0; kb < p.nkb; ++kb, ++pos) {
          const int s = (int)(pos % kStages);
          const uint32_t ph = (uint32_t)((pos / kStages) & 1);
          if (!mbar_wait(full(s), ph, p.wait_polls, p.wait_ns)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = d0 + (p.fp8 ? (uint32_t)(kb * TI) : 0u);
          for (int kk = 0; kk < 4; ++kk) {   // 4 MMAs of 32 bytes of K each
            const uint64_t a = sdesc_sw128(sOpA + s * kStageA + kk * 32);
            const uint64_t b = sdesc_sw128(sOpB + s * kStageB + kk * 32);
            const uint32_t acc = p.fp8 ? (kk > 0) : (kb > 0 || kk > 0);
            if constexpr (kPair) {
              tc_mma_f16_pair(d, a, b, idesc, acc);
            } else {
              if (p.fp8) tc_mma_f8(d, a, b, idesc, acc);
              else tc_mma_f16(d, a, b, idesc, acc);
            }
          }
          commit(empty(s));   // the stage is free once these MMAs have read it
        }
        commit(acc_full(ab));
      }
      if (!ok) atomicOr(p.status, kErrTimeout);
      // every MMA issued has completed before TMEM is freed, also when an
      // epilogue group gave up before the last accumulator was written
      commit(mma_drain);
      if (!mbar_wait(mma_drain, 0)) atomicOr(p.status, kErrTimeout);
      if constexpr (kPair) report_end(2, pos);
    }
  } else if (Cfg::kMover && warp >= 2 + kEpiGroups * kEpiWarps) {
    // C mover of group g: a segment's C is loaded ahead of the epilogue, and
    // stored and replaced by that of the buffer's next tile as soon as the
    // epilogue is done with that segment, so that the round trip (store read,
    // load) of one segment passes while the other is worked on.  With the group's
    // leader moving whole tiles, the one buffer of a 256-row tile was the bound up
    // to a depth of 512: C -= A B of order 16384, depth 256: 324 -> 228 us, depth
    // 512: 316 -> 275 (what is left there is the operands' intake, 48 KB per 64
    // of depth); order 28672, depth 512: 892 -> 880.  (With three buffers the trip
    // is hidden anyway and the hop to the mover costs: see the epilogue.)
    if (lane == 0 && p.has_c) {
      const int g = warp - 2 - kEpiGroups * kEpiWarps;
      int loading[kSegs];   // the phase of a load whose segment the epilogue has not finished, or -1
      auto arm = [&](const TileLoc& L, int h, uint32_t phase) {
        if (!load_c) {
          mbar_arrive(c_full(0, g, h));
          return;
        }
        loading[h] = (int)phase;
        load_c_seg(L, 0, g, h);
      };
      acquire_maps(2);
#pragma unroll
      for (int h = 0; h < kSegs; ++h) {
        loading[h] = -1;
        if (first() < p.ntiles) arm(locate(first()), h, 0);
      }
      bool ok = true;
      uint32_t phase = 0;
      for (int t = first(); t < p.ntiles && ok; t += stride(), phase ^= 1) {
        const TileLoc L = locate(t);
#pragma unroll 1
        for (int h = 0; h < kSegs; ++h) {
          if (!mbar_wait(c_done(0, g, h), phase, p.wait_polls, p.wait_ns)) { ok = false; break; }
          loading[h] = -1;
          if (!kPair || L.j0 < L.N) store_c_seg(L, 0, g, h);
          bulk_commit();
          const int t2 = t + stride();
          if (t2 < p.ntiles) {
            asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            arm(locate(t2), h, phase ^ 1);
          }
        }
      }
      bulk_wait0();
      if (!ok) {
        atomicOr(p.status, kErrTimeout);
        // C loads that the epilogue did not reach land before the CTA exits
        for (int h = 0; h < kSegs; ++h)
          if (loading[h] >= 0) mbar_wait(c_full(0, g, h), (uint32_t)loading[h]);
      }
    }
  } else {
    // epilogue: group g = (warp - 2) / 4 owns rows i0 + (TI/2) g .. + TI/2 - 1 of the
    // tile, as kSegs segments of 64 rows; thread = output column j = j0 + jl,
    // jl = 32 q + lane (its TMEM lane)
    const int q = warp & 3;
    const int g = (warp - 2) >> 2;
    const int jl = 32 * q + lane;
    // Three buffers: the group's first thread moves its C.  The C of the tile after next is loaded into
    // the buffer of the tile before this one once this one's store has been issued, by when that store
    // has been read, so that the group never waits for its own.  A warp that moves it instead costs
    // these short tiles more than the group's barriers do (C = A B of order 16384, depth 128: 216 us
    // with it, 181 without; C -= A B of order 24000: 517 and 501).
    const bool leader = !Cfg::kMover && p.has_c && ((warp - 2) & 3) == 0 && lane == 0;
    int loading[kCBufs];   // (leader) the phase of a load whose tile the group has not reached, or -1
#pragma unroll
    for (int b = 0; b < kCBufs; ++b) loading[b] = -1;
    auto load_ahead = [&](int t, int b, int phase) {
      if (!load_c || t >= p.ntiles) return;
#pragma unroll
      for (int k = 0; k < kCBufs; ++k) loading[k] = k == b ? phase : loading[k];
      load_c_seg(locate(t), b, g, 0);
    };
    if (leader) {
      acquire_maps(2);
#pragma unroll
      for (int b = 0; b < kCBufs - 1; ++b) load_ahead(first() + b * stride(), b, 0);
    }
    bool ok = true;
    int local = 0;
    for (int t = first(); t < p.ntiles && ok; t += stride(), ++local) {
      const TileLoc L = locate(t);
      const int i0 = L.i0, j0 = L.j0;
      const int cb = local % kCBufs, ab = local % p.nbuf;
      const uint32_t cphase = (uint32_t)((local / kCBufs) & 1);
      // One decision per warp (uniform for tcgen05.ld); a warp that gives up leaves its segment undone,
      // which the mover's and the other waits run out on.  Without a mover one per group, whose warps
      // meet at its barriers; this one also says that the buffer's last store has been read.
      ok = !(Cfg::kMover ? p.has_c : load_c) || mbar_wait(c_full(cb, g, 0), cphase, p.wait_polls, p.wait_ns);
      ok = ok && mbar_wait(acc_full(ab), (uint32_t)((local / p.nbuf) & 1), p.wait_polls, p.wait_ns);
      ok = Cfg::kMover ? __all_sync(0xffffffffu, ok) : epi_all(g, ok);
      if (!ok) break;
      if (leader) {
#pragma unroll
        for (int k = 0; k < kCBufs; ++k) loading[k] = k == cb ? -1 : loading[k];
      }
      tc_fence_after();
      const uint32_t lane_base = tmem + (uint32_t)ab * p.acc_cols + ((uint32_t)(32 * q) << 16) + (TI / 2) * g;
      float sc[4] = {1.0f, 1.0f, 1.0f, 1.0f};
      if (p.fp8)
        for (int s2 = 0; s2 < p.nkb && s2 < 4; ++s2)
          sc[s2] = __fmul_rn(p.sA[(i0 / 128) * p.sa_ld + s2], p.sB[(j0 / 128) * p.sb_ld + s2]);
      const int64_t j = (int64_t)j0 + jl;
#pragma unroll 1
      for (int h = 0; h < kSegs; ++h) {   // 64-row segments of the group's rows
        if (h > 0 && p.has_c) {
          ok = __all_sync(0xffffffffu, mbar_wait(c_full(cb, g, h), cphase, p.wait_polls, p.wait_ns));
          if (!ok) break;
        }
        const uint32_t lane_addr = lane_base + 64u * h;
        float acc[64];
        {
          uint32_t r[64];
          if (p.fp8) {
#pragma unroll
            for (int v = 0; v < 64; ++v) acc[v] = 0.0f;
            for (int s2 = 0; s2 < p.nkb; ++s2) {
              tmem_ld64(lane_addr + (uint32_t)(s2 * TI), r);
#pragma unroll
              for (int v = 0; v < 64; ++v) acc[v] = __fmaf_rn(__uint_as_float(r[v]), sc[s2], acc[v]);
            }
          } else {
            tmem_ld64(lane_addr, r);
#pragma unroll
            for (int v = 0; v < 64; ++v) acc[v] = __uint_as_float(r[v]);
          }
        }
        if (h == kSegs - 1) {
          // accumulator buffer free for the MMA warp as soon as it is in registers
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            if (kPair && rank == 1) mbar_arrive_cluster(smem_at(acc_empty(ab), 0));
            else mbar_arrive(acc_empty(ab));
          }
        }
        if constexpr (CB == 4) {
          // fp32 C: two 32-row boxes; rows 32 q + 4 c8 .. +3 of column j in chunk c8 of box q
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const uint32_t row_addr = sC + cb * kCTile + (g * kBoxes + 2 * h + q) * kCBox + jl * 128;
#pragma unroll
            for (int c8 = 0; c8 < 8; ++c8) {
              const uint32_t ad = row_addr + ((c8 ^ (jl & 7)) << 4);
              float cf[4];
              asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                           : "=f"(cf[0]), "=f"(cf[1]), "=f"(cf[2]), "=f"(cf[3]) : "r"(ad) : "memory");
#pragma unroll
              for (int v = 0; v < 4; ++v) cf[v] = __fsub_rn(cf[v], acc[32 * q + 4 * c8 + v]);
              asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};"
                           ::"r"(ad), "f"(cf[0]), "f"(cf[1]), "f"(cf[2]), "f"(cf[3]) : "memory");
            }
          }
        } else {
        // rows i0 + (TI/2) g + 64 h + 8 ch .. +7 of column j: eight 16-byte chunks of the swizzled box
        const uint32_t cbox = sC + cb * kCTile + (g * kBoxes + h) * kCBox;
        const uint32_t row_addr = cbox + jl * 128;
#pragma unroll
        for (int ch = 0; ch < 8; ++ch) {
          const uint32_t ad = row_addr + ((ch ^ (jl & 7)) << 4);
          uint32_t outw[4];
          if (p.mode == kEpiSub) {
            uint32_t cw[4];
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(cw[0]), "=r"(cw[1]), "=r"(cw[2]), "=r"(cw[3]) : "r"(ad) : "memory");
#pragma unroll
            for (int v = 0; v < 4; ++v) {
              const float lo = __fsub_rn(u16_to_f32((uint16_t)(cw[v] & 0xffffu), p.fmt), acc[8 * ch + 2 * v]);
              const float hi = __fsub_rn(u16_to_f32((uint16_t)(cw[v] >> 16), p.fmt), acc[8 * ch + 2 * v + 1]);
              outw[v] = pack16x2(lo, hi, p.fmt);
            }
          } else {
#pragma unroll
            for (int v = 0; v < 4; ++v)
              outw[v] = pack16x2(p.sign * acc[8 * ch + 2 * v], p.sign * acc[8 * ch + 2 * v + 1], p.fmt);
          }
          if (p.has_c)
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                         ::"r"(ad), "r"(outw[0]), "r"(outw[1]), "r"(outw[2]), "r"(outw[3]) : "memory");
          if (L.R && j < L.N) {
#pragma unroll
            for (int v = 0; v < 8; ++v) {
              const int64_t i = (int64_t)i0 + (TI / 2) * g + 64 * h + 8 * ch + v;
              if (i < L.M) L.R[i * L.ldr + j] = (uint16_t)((outw[v >> 1] >> ((v & 1) * 16)) & 0xffffu);
            }
          }
        }
        }
        if (p.has_c) {
          fence_async_smem();
          if constexpr (Cfg::kMover) {
            __syncwarp();
            if (lane == 0) mbar_arrive(c_done(cb, g, h));
          } else {
            epi_all(g, true);
            if (leader) {
              store_c_seg(L, cb, g, 0);
              bulk_commit();
              asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
              const int ahead = local + kCBufs - 1;
              load_ahead(t + (kCBufs - 1) * stride(), ahead % kCBufs, (ahead / kCBufs) & 1);
            }
          }
        }
      }
    }
    if (!ok && lane == 0) atomicOr(p.status, kErrTimeout);
    if (leader) {
      bulk_wait0();
      // C loads that the group did not reach land before the CTA exits
#pragma unroll
      for (int b = 0; b < kCBufs; ++b)
        if (loading[b] >= 0 && !mbar_wait(c_full(b, g, 0), (uint32_t)loading[b])) atomicOr(p.status, kErrTimeout);
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (kPair) {
    // neither CTA of a pair leaves while the other may still read its shared memory or arrive there
    cluster_sync();
    if (ended[0] != ended[1] || ended[0] != ended[2]) {
      // A wait ran out (the same three values, so the same decision in both CTAs).  A stage loaded by
      // one rank only would never complete on rank 0's barrier: the other rank loads it too.  The stage
      // is free there, since the MMAs before it released both CTAs' together.  Then rank 0 waits for all.
      const int most = max(ended[0], ended[1]);
      if (threadIdx.x == 0) {
        for (int pos = ended[rank]; pos < most; ++pos) load_stage(locate(first() + pos / p.nkb * stride()), pos % p.nkb, pos);
        if (rank == 0) drain_loads(most);
      }
      __syncthreads();
      cluster_sync();
    }
    // rank 0's last commit arrives here too
    if (rank == 1 && threadIdx.x == 32 && !mbar_wait(mma_drain, 0)) atomicOr(p.status, kErrTimeout);
    __syncwarp();
  }
  if (warp == 1) {
    tc_fence_after();
    if constexpr (kPair) tmem_dealloc_pair(tmem, p.ncols);
    else tmem_dealloc(tmem, p.ncols);
  }
  if (p.span && threadIdx.x == 0) atomicMin(p.span + 1, ~global_ns());
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  });
  return fn;
}

// 2-D map over 16-bit (or, with u32, 32-bit) units: `rows` rows of `inner`
// units, consecutive rows `ld_bytes` apart, box = box_inner x box_rows,
// 128-byte swizzle, zero fill outside the matrix.
bool make_map(CUtensorMap* tm, const void* base, uint64_t inner, uint64_t rows, uint64_t ld_bytes,
              uint32_t box_inner, uint32_t box_rows, bool u32 = false) {
  auto fn = encode_fn();
  if (!fn) return false;
  if (((uintptr_t)base & 15) || (ld_bytes & 15) || inner == 0 || rows == 0) return false;
  cuuint64_t dims[2] = {inner, rows};
  cuuint64_t strides[1] = {ld_bytes};
  cuuint32_t box[2] = {box_inner, box_rows};
  cuuint32_t es[2] = {1, 1};
  return fn(tm, u32 ? CU_TENSOR_MAP_DATA_TYPE_UINT32 : CU_TENSOR_MAP_DATA_TYPE_UINT16, 2, const_cast<void*>(base),
            dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}


int num_sms() {
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 148;
  }
  return sms;
}

// persistent grid size: the SM count, or the calling thread's SM budget
int grid_cap() {
  const int b = sm_budget();
  return b > 0 ? std::min(b, num_sms()) : num_sms();
}

}  // namespace

namespace {

template <int TI, int CB = 2, bool kPair = false>
cudaError_t gemm_tc_tiles(const GemmArgs& g, cudaStream_t st, const GemmArgs* also = nullptr) {
  using Cfg = TileCfg<TI, CB, kPair>;
  static_assert(CB == 2 || TI == 128, "fp32 C on 128-row tiles only");
  if (CB == 4 && (g.mode != kEpiSub || g.R || !g.C)) return cudaErrorInvalidValue;
  const int esz = g.fp8 ? 1 : 2;
  const uint64_t kbytes = (uint64_t)g.K * esz;
  if (kbytes % kRowBytes) return cudaErrorInvalidValue;
  CUtensorMap ta, tb, tc;
  if (!make_map(&ta, g.A, kbytes / 2, (uint64_t)g.M, (uint64_t)g.lda * esz, kRowBytes / 2, Cfg::kRowsB) ||
      !make_map(&tb, g.B, kbytes / 2, (uint64_t)g.N, (uint64_t)g.ldb * esz, kRowBytes / 2, kTJ))
    return cudaErrorInvalidValue;
  TcParams p{};
  p.has_c = g.C != nullptr;
  if (p.has_c) {
    // column-major C: inner = rows; box = 128 bytes of rows (64 16-bit or 32 fp32) x 128 columns
    if (!make_map(&tc, g.C, (uint64_t)g.M, (uint64_t)g.N, (uint64_t)g.ldc * CB, Cfg::kBoxRows, kTJ, CB == 4))
      return cudaErrorInvalidValue;
  } else {
    tc = ta;   // never dereferenced
  }
  p.M = g.M; p.N = g.N; p.nkb = (int)(kbytes / kRowBytes);
  p.tiles_i = cdiv(g.M, TI);
  p.ntiles = p.tiles_i * cdiv(g.N, (kPair ? 2 : 1) * kTJ);
  p.split = p.ntiles;
  TcSecond second{};
  if (also) {
    const GemmArgs& h = *also;
    if (h.fp8 || h.c32 || h.K != g.K || h.mode != g.mode || h.sign != g.sign || h.fmt != g.fmt || !h.C || !g.C ||
        !make_map(&second.a, h.A, kbytes / 2, (uint64_t)h.M, (uint64_t)h.lda * esz, kRowBytes / 2, TI) ||
        !make_map(&second.b, h.B, kbytes / 2, (uint64_t)h.N, (uint64_t)h.ldb * esz, kRowBytes / 2, kTJ) ||
        !make_map(&second.c, h.C, (uint64_t)h.M, (uint64_t)h.N, (uint64_t)h.ldc * CB, Cfg::kBoxRows, kTJ, CB == 4))
      return cudaErrorInvalidValue;
    second.M = h.M; second.N = h.N; second.tiles_i = cdiv(h.M, TI);
    second.R = (uint16_t*)h.R; second.ldr = h.ldr;
    p.ntiles += second.tiles_i * cdiv(h.N, kTJ);
  }
  p.mode = g.mode; p.sign = g.sign; p.fmt = g.fmt; p.fp8 = g.fp8;
  p.R = (uint16_t*)g.R; p.ldr = g.ldr;
  p.sA = g.sA; p.sa_ld = g.sa_ld; p.sB = g.sB; p.sb_ld = g.sb_ld;
  p.status = g.status;
  const WaitBudget wb = wait_budget();
  p.wait_polls = wb.polls;
  p.wait_ns = wb.ns;
  if (g.fp8) {
    if (TI != 128 || p.nkb > 4) return cudaErrorInvalidValue;   // one 128-column accumulator per slice
    p.acc_cols = (uint32_t)(TI * p.nkb);
  } else {
    p.acc_cols = TI;
  }
  p.nbuf = (2 * p.acc_cols <= 512u) ? 2 : 1;
  uint32_t need = p.acc_cols * (uint32_t)p.nbuf, ncols = 32;
  while (ncols < need) ncols <<= 1;
  p.ncols = ncols;

  static std::atomic<int> configured_for{-1};
  int dev = 0;
  cudaGetDevice(&dev);
  if (configured_for.load() != dev) {
    cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<TI, CB, kPair>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Cfg::kSmem);
    if (e != cudaSuccess) return e;
    configured_for.store(dev);
  }
  const int cap = g.max_ctas > 0 ? std::min(g.max_ctas, grid_cap()) : grid_cap();
  const int grid = kPair ? 2 * std::min(p.ntiles, cap / 2) : std::min(p.ntiles, cap);
  // algorithmic DRAM bytes: both operands once, C read (subtract mode) and
  // written once, the optional row-major copy written once
  double flops = 0.0, bytes = 0.0;
  for (const GemmArgs* h : {&g, also}) {
    if (!h) continue;
    const double mn = (double)h->M * (double)h->N;
    flops += 2.0 * mn * h->K;
    bytes += ((double)h->M + (double)h->N) * (double)h->K * esz +
             (p.has_c ? mn * CB * (h->mode == kEpiSub ? 2.0 : 1.0) : 0.0) + (h->R ? mn * 2.0 : 0.0);
  }
  void* tok = prof_begin(st);
  p.span = prof_device_span(tok);
  const cudaError_t e =
      launch_pdl_cluster(gemm_tc_kernel<TI, CB, kPair>, kPair ? 2 : 1, dim3(grid), dim3(Cfg::kThreads), Cfg::kSmem,
                         st, ta, tb, tc, p, (const GemmGroupItem*)nullptr, 0, second);
  prof_end(tok, g.mode == kEpiSub ? kProfGemm : kProfGemmStore, flops, st, bytes);
  count_launches(1);
  return e;
}

}  // namespace

bool encode_f64_map(CUtensorMap* tm, const double* base, int64_t rows, int64_t cols, int64_t ld, int box_rows,
                    int box_cols) {
  auto fn = encode_fn();
  if (!fn || ((uintptr_t)base & 15) || (ld & 1)) return false;
  cuuint64_t dims[2] = {(cuuint64_t)rows, (cuuint64_t)cols};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 8};
  cuuint32_t box[2] = {(cuuint32_t)box_rows, (cuuint32_t)box_cols};
  cuuint32_t es[2] = {1, 1};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<double*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool gemm_group_encode(const GemmArgs* gs, int count, GemmGroupItem* items, int* total_tiles) {
  static_assert(sizeof(CUtensorMap) == 128, "tensor map size");
  int tiles = 0;
  for (int c = 0; c < count; ++c) {
    const GemmArgs& g = gs[c];
    if (g.fp8 || g.c32 || g.K <= 0 || g.K >= 256 || (g.K % 128) || g.K != gs[0].K || g.mode != gs[0].mode ||
        !g.C || g.M <= 0 || g.N <= 0)
      return false;
    const uint64_t kbytes = (uint64_t)g.K * 2;
    CUtensorMap* ta = reinterpret_cast<CUtensorMap*>(items[c].maps[0]);
    CUtensorMap* tb = reinterpret_cast<CUtensorMap*>(items[c].maps[1]);
    CUtensorMap* tc = reinterpret_cast<CUtensorMap*>(items[c].maps[2]);
    if (!make_map(ta, g.A, kbytes / 2, (uint64_t)g.M, (uint64_t)g.lda * 2, kRowBytes / 2, 128) ||
        !make_map(tb, g.B, kbytes / 2, (uint64_t)g.N, (uint64_t)g.ldb * 2, kRowBytes / 2, kTJ) ||
        !make_map(tc, g.C, (uint64_t)g.M, (uint64_t)g.N, (uint64_t)g.ldc * 2, 64, kTJ))
      return false;
    items[c].M = g.M;
    items[c].N = g.N;
    items[c].tiles_i = cdiv(g.M, 128);
    items[c].tile_begin = tiles;
    items[c].R = g.R;
    items[c].ldr = g.ldr;
    tiles += items[c].tiles_i * cdiv(g.N, kTJ);
  }
  *total_tiles = tiles;
  return true;
}

cudaError_t gemm_tc_grouped(const GemmArgs& g, const GemmGroupItem* dev_items, int nitems, int total_tiles,
                            cudaStream_t st, double flops, double bytes) {
  using Cfg = TileCfg<128, 2>;
  if (nitems <= 0 || total_tiles <= 0) return cudaSuccess;
  TcParams p{};
  p.has_c = 1;
  p.nkb = (int)((uint64_t)g.K * 2 / kRowBytes);
  p.tiles_i = 1;
  p.ntiles = p.split = total_tiles;
  p.mode = g.mode; p.sign = g.sign; p.fmt = g.fmt; p.fp8 = 0;
  p.status = g.status;
  const WaitBudget wb = wait_budget();
  p.wait_polls = wb.polls;
  p.wait_ns = wb.ns;
  p.acc_cols = 128;
  p.nbuf = 2;
  p.ncols = 256;
  static std::atomic<int> configured_for{-1};
  int dev = 0;
  cudaGetDevice(&dev);
  if (configured_for.load() != dev) {
    cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<128, 2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Cfg::kSmem);
    if (e != cudaSuccess) return e;
    configured_for.store(dev);
  }
  const int grid = std::min(total_tiles, g.max_ctas > 0 ? std::min(g.max_ctas, grid_cap()) : grid_cap());
  CUtensorMap none;
  memset(&none, 0, sizeof(none));   // the items' maps are used instead
  void* tok = prof_begin(st);
  p.span = prof_device_span(tok);
  const cudaError_t e = launch_pdl(gemm_tc_kernel<128, 2, false>, dim3(grid), dim3(Cfg::kThreads), Cfg::kSmem, st, none, none,
                                   none, p, dev_items, nitems, TcSecond{});
  prof_end(tok, g.mode == kEpiSub ? kProfGemm : kProfGemmStore, flops, st, bytes);
  count_launches(1);
  return e;
}

namespace {

// A tile height of 128 (hpmxp_set_tuning or HPMXP_GEMM_TILE=128) keeps every
// product on the 128-row tile.
bool wide_tiles_enabled() { return tuning().gemm_tile != 128; }

}  // namespace

cudaError_t gemm_tc(const GemmArgs& g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  if (g.c32) return g.fp8 ? cudaErrorInvalidValue : gemm_tc_tiles<128, 4>(g, st);
  // 256-row tiles for the 16-bit products that fill them (M >= 256) and have
  // enough depth (K >= 256) for one C buffer to keep up
  if (!g.fp8 && g.M >= 256 && g.K >= 256 && wide_tiles_enabled()) {
    // Pairs of CTAs where the operands' intake is the bound: a depth of 512 and
    // more tiles than SMs.  Pairs / single CTAs, C -= A B, us: order 28672, depth
    // 512: 710 / 884; 16384: 245 / 284; 8192: 80 / 93; 3072: 28.5 / 30.3; 2048
    // (fewer tiles than SMs): 25.7 / 25.1; depth 384 at 16384: 246 / 241; depth
    // 256 at 28672: 699 / 687 (the C round trip bounds both).  An odd number of
    // 128-column tiles leaves half of the last pairs empty, which pays from seven
    // on: 30000 rows, 128 columns (a panel's) 35.5 / 28.5; 384: 34.3 / 32.5; 512:
    // 33.4 / 36.0; 640: 38.6 / 37.7; 896: 46.6 / 49.1.
    const int cap = g.max_ctas > 0 ? std::min(g.max_ctas, grid_cap()) : grid_cap();
    const int jt = cdiv(g.N, kTJ);
    if (g.K >= 512 && cap >= 2 && (jt % 2 == 0 || jt >= 7) && (long long)cdiv(g.M, 256) * jt > num_sms())
      return gemm_tc_tiles<256, 2, true>(g, st);
    return gemm_tc_tiles<256>(g, st);
  }
  return gemm_tc_tiles<128>(g, st);
}

// Two independent 16-bit products of the same depth in one launch, on 128-row
// tiles (either may be empty).
cudaError_t gemm_tc_pair(const GemmArgs& g, const GemmArgs& h, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0) return gemm_tc(h, st);
  if (h.M <= 0 || h.N <= 0) return gemm_tc(g, st);
  return gemm_tc_tiles<128>(g, st, &h);
}

}  // namespace hpmxp
