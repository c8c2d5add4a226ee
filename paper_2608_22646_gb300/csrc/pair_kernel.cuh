// LM head of the multi-kernel step, on CTA pairs (tcgen05 cta_group::2): the
// same quantities as lm_head_softmax_kernel (Box 1 of arXiv 2608.22646:
// c_i = max_v p_theta(x_i = v) and argmax_v p_theta, logits never leaving
// tensor memory), for any number M >= 1 of masked rows, in one of two
// orientations chosen per step from M (pair_swapped).
//
// Unswapped, for wide steps: with hundreds to thousands of rows the
// contraction is tensor-bound (2 V H M flops against 2 V H bytes of W), so
// the masked rows fill the MMA M dimension and the vocabulary the N
// dimension.  One tcgen05.mma of the pair computes a 256 x 256 tile: each CTA
// holds 128 of the rows (its A half) and 128 of the vocabulary rows (its B
// half) per K block, and keeps its 128 x 256 half of the accumulator in
// tensor memory.  Per K block a CTA loads 32 KiB (16 KiB of hidden rows,
// 16 KiB of W) for 2 * 128 * 256 * 64 flops, half the shared-memory traffic
// per flop of a single-CTA 128 x 256 tile.  A tensor-memory lane holds one
// row's logits, so the epilogue is a serial online softmax per thread, no
// shuffles; two warps share a row's columns.
//
// Swapped, for narrow steps: the vocabulary fills the MMA M dimension (256
// rows per pair, 128 per CTA: the W half is the A operand) and the masked
// rows the N dimension.  The M rows are split into n_rt = ceil(M / 256) row
// tiles of equal width N (a multiple of 32, at most 256), so a step pads at
// most 31 rows per tile instead of up to 255: M = 305 runs as two 160-column
// tiles, M = 159 as one of 160, M = 5 as one of 32.  A tensor-memory lane
// then holds one vocabulary row of every column; the epilogue reads fragments
// in which a thread holds four vocabulary rows of a column, folds them into a
// running triple per column over all of the pair's tiles, and merges across
// lanes and warps once, at the end (every tile, when a pair's tiles have
// different row tiles).  Each CTA writes the triples of its half of the
// vocabulary rows: two partials per pair.  Each CTA loads N / 2 of a tile's
// rows per K block as one box of exactly that many rows.  A step runs swapped
// when N is at most swap_max_n (by default pair_swap_width(H)).
//
// The epilogue of a pair's last tile is not hidden by anything.  With one warp
// per quarter and a 31-merge transposition per tile it took 6 us at N = 96 and
// 12 us at N = 192 after the last copy, and it bounded whole steps of models
// with a short K (22000 x 1024, M = 192: 37.4 us a step, now 25.7; M = 352
// 48.1 -> 27.9; unswapped M = 224 27.9 -> 21.9).  At 4096 x 126464 a step takes
// 165.8 us instead of 172.5 at M = 192, 245 instead of 254.6 at M = 352 (these
// with the set-up below).
//
// Partials: when the number of pairs is a multiple of the number of row
// tiles n_rt, every tile of a pair has the same row tile, and the epilogue
// folds its tiles into one partial (max * log2 e, sum of 2^(z log2 e - max),
// argmax) per row and pair (and CTA, swapped), which the commit reads
// directly (pair_partials_per_row); otherwise it writes one partial per row
// and vocabulary tile (and CTA), merged per row by reduce_partials_kernel.
//
// Work: tiles (v, j) of 256 vocabulary rows x one row tile, numbered
// t = v * n_rt + j and dealt round-robin to the pairs of a persistent grid.
// The pairs working at one time share few W tiles, each read from HBM once
// and by the n_rt pairs of its row tiles from L2; the gathered hidden rows
// (at most 2 x 65536 x 16384 bytes, in practice tens of MB) stay in L2.
//
// Roles per CTA (320 threads): warp 0 producer (hidden half and W half by
// TMA; W from a packed copy in which every box is one contiguous block, or
// kStatic from the caller's rows); warp 1 allocates tensor memory and, in the
// even CTA, issues the MMAs; warps 2..9 epilogue.  Both CTAs' copies of a stage complete on
// the even CTA's barrier (cta_group::2 loads), which the even CTA's producer
// arms with the bytes of both.  Two accumulator buffers let the epilogue of
// one tile overlap the next tile's MMAs.  Barriers, tensor memory and map
// prefetches come before the dependency wait, so that a step's first copies
// start right after the gather.
//
// How stages are issued.  The producer and the MMA warp run their loops with
// all 32 lanes, every loop bound and descriptor the same in each, and only the
// issuing instructions are predicated on one elected lane: the descriptors and
// coordinates then stay in uniform registers, where the TMA and MMA
// instructions take them from.  With the loops inside `if (lane == 0)` each
// MMA cost its thread ~50 ns and a stage 300 ns whatever its width, more than
// its copies and its tensor work.  Measured, 4096 x 126464, one step's head:
// M = 264 269 -> 209 us, M = 352 279 -> 238 us, M = 512 297 -> 286 us,
// M = 2048 1.09 -> 1.04 ms, M = 128 165 -> 157 us; of it, the MMA warp alone
// gave 42 us at M = 264 and the producer 17 us.  A wait that gives up makes its
// lane stop waiting and issuing, not leave the loop, so that no vote is needed
// per stage (a vote costs 1 to 4 us a step); the warp leaves together at the
// end of the tile.
//
// What bounds a step: reading W from HBM with one row tile.  With two narrow
// ones, filling the stages from L2 (26 KiB per CTA and 250 ns at N = 160, every
// CTA at once); with wide ones the tensor cores.  A second issuing thread
// would run MMAs side by side, but two threads accumulating into one
// accumulator do so in no fixed order, and the fp32 logits (and the commit
// decisions at a threshold) would then change from run to run.
#pragma once

#include <climits>
#include "head_kernel.cuh"
#include "ptx.cuh"
#include "softmax.cuh"

namespace cai {

constexpr int kPairEpiWarps = 8;      // two per tensor-memory quarter, half of the columns each
constexpr int kPairThreads = 64 + 32 * kPairEpiWarps;
// Registers a thread.  No spills at 160, and a block takes the same time at 168
// (66 to 512 rows, five shapes).  They do not decide what fits beside a pair
// CTA: with the exchange buffer of swapped contexts its shared memory leaves the
// SM to nothing else, and a commit CTA (512 threads) would not fit either way.
constexpr int kPairRegs = 160;
constexpr int kPairTileRows = 256;    // masked rows per pair tile (MMA M)
constexpr int kPairTileVocab = 256;   // vocabulary rows per pair tile (MMA N)
constexpr int kPairHalf = 128;        // rows of each per CTA
constexpr int kPairBlockK = 64;       // K per stage (one 128-byte swizzled row)
constexpr int kPairHalfBytes = kPairHalf * kPairBlockK * 2;  // 16 KiB
constexpr int kPairStageBytes = 2 * kPairHalfBytes;          // A half + B half
constexpr int kPairTmemCols = 2 * kPairTileVocab;            // two accumulators
constexpr int kSwapTwoBlocks = 96;  // swapped tiles up to this wide: two K blocks per stage
constexpr int kSwapColStep = 32;    // swapped orientation: granularity of N
constexpr int kSwapXchBytes = 2 * 4 * kPairTileVocab * 16;  // cross-warp exchange, two buffers
constexpr int kSwapChunks = kPairTileVocab / 32;  // most 16-column chunks of an epilogue warp
constexpr int kPairMaxRing = 12;    // swapped stages are cut to size: up to this many

// Tensor maps of the gathered rows with boxes of 16, 32, ..., 128 rows
// (swapped orientation: a CTA's N / 2 rows of a tile, a multiple of 16, load
// as one exact box: each TMA copy has a fixed cost, and every byte written
// to shared memory competes with the MMAs' operand reads).
struct PairRowMaps {
  CUtensorMap box[8];  // box[q]: 16 (q + 1) rows
};

struct PairParams {
  const int* d_M;      // masked rows of this step (device)
  int* m_hist_slot;    // where this step's M is recorded, or null
  float4* part;        // [rows, n_vt] partial per row and vocabulary tile
  uint32_t* err;
  int V, H;
  int n_vt;            // ceil(V / 256)
  int min_M;           // smaller steps are left to lm_head_softmax_kernel (<= 1: this
                       // kernel decodes every step and records M = 0 too)
  int swap_max_n;      // steps whose swapped tile width is at most this run swapped
  int n_stages;
  const float* inv_r;  // final-norm row scales [rows] (kNorm only)
  int ring_max;        // most stages in flight (<= kPairMaxRing)
  int M_fixed;         // kStatic: rows of this launch
  int th1, n_vt1;      // steps of one row tile: vocabulary rows per CTA and tile, tiles
  // W map coordinates of K block kb, vocabulary row r (a tile's first): (kb w_dx, r w_ry + kb w_dy).
  int w_dx, w_dy, w_ry;
};

// Row tiles of a pair step with M rows (both orientations).
__host__ __device__ inline int pair_row_tiles(int M) {
  return (M + kPairTileRows - 1) / kPairTileRows;
}

// Swapped orientation: width N of each of the n_rt row tiles; tile j covers
// rows [j N, j N + N), the last one possibly past M (padding, never written).
__host__ __device__ inline int swap_tile_cols(int M, int n_rt) {
  const int per = (M + n_rt - 1) / n_rt;
  return (per + kSwapColStep - 1) / kSwapColStep * kSwapColStep;
}

// Orientation of a pair step with M rows: swapped when the tile width of the
// swapped orientation is at most swap_max_n (0: never).
__host__ __device__ inline bool pair_swapped(int M, int swap_max_n) {
  return M > 0 && swap_tile_cols(M, pair_row_tiles(M)) <= swap_max_n;
}

// Widest swapped tile by default, from the length of the contraction: the
// swapped orientation pads fewer rows, but its epilogue takes longer per tile,
// and the shorter K is the less of it is hidden.  0: always unswapped.
// Measured, microseconds a step, swapped against unswapped: H = 256 (V = 4096)
// N = 32 13.7 / 12.6; H = 512 (22000) N = 64 17.4 / 17.5, N = 96 18.5 / 17.6;
// H = 1024 (50003) N = 96 27.2 / 28.5, N = 160 29.9 / 28.8; H = 2048 (50003)
// N = 192 48.3 / 46.3, two tiles of 160 57.5 / 66.5; H = 4096 (126464) N = 224
// 171 / 172, two tiles of 224 271 / 299, N = 256 183 / 182.  One limit serves
// steps of one tile and of several, whose gain is the larger: at H = 2048 the
// single tiles of 192 lose 2 us so that two tiles of that width win.
__host__ __device__ inline int pair_swap_width(int H) {
  return H < 384 ? 0 : H < 768 ? 64 : H < 1536 ? 96 : H < 3072 ? 192 : 224;
}

// Partials per row written by a pair step with M rows on n_pairs pairs: one
// per pair of the row's tile (two in the swapped orientation, one per CTA)
// when n_pairs is a multiple of the row-tile count, else 0 (one per
// vocabulary tile, two when swapped, merged by the reduce kernel).
__host__ __device__ inline int pair_partials_per_row(int M, int n_pairs, bool swap) {
  const int n_rt = pair_row_tiles(M);
  if (n_rt <= 0 || n_pairs % n_rt != 0) return 0;
  return (swap ? 2 : 1) * (n_pairs / n_rt);
}

// Vocabulary rows per CTA and tile of a step of one row tile: such a step is
// bound by reading W, so V is dealt out evenly, every pair the same number n
// of tiles of equal height (a multiple of 8 rows, the swizzle atom, at most
// 128).
__host__ __device__ inline int pair_even_rows(int V, int n_pairs) {
  const int n = (V + 2 * kPairHalf * n_pairs - 1) / (2 * kPairHalf * n_pairs);
  const int per = (V + 2 * n_pairs * n - 1) / (2 * n_pairs * n);
  return (per + 7) / 8 * 8;
}

// ... of a context, whose packed W then has the matching order (pair_w_run).
// From five tiles a pair on, 128-row tiles are kept: pairs that finish early
// leave their share of the memory bandwidth to the others, and the order that
// even tiles need reads 128-row tiles a little slower.  Measured, microseconds
// a step: 22000 x 1024 (n = 2), M = 224 28.3 -> 25.5 with even tiles; 126464 x
// 4096 (n = 7), M = 128 165.7 -> 163.8, but M = 264 232.7 -> 236.
__host__ __device__ inline int pair_tile_rows(int V, int n_pairs) {
  return V > 4 * 2 * kPairHalf * n_pairs ? kPairHalf : pair_even_rows(V, n_pairs);
}

// Whether W is read evict-first (kFirst, contexts of up to two row tiles).  A
// weight well above what L2 keeps is better not kept: what stays is then an
// unbroken part of it that the next step finds (1024 x 64000, M = 160: 35.9 ->
// 32.7 us a step; 2048 x 50003 47.3 -> 43.6; 4096 x 126464 161.5 -> 158.2), a
// smaller one is (1024 x 40000, 26.6 us, 27.2 evict-first).  Read in place from
// row-major W the line lies higher: 1024 x 50003, 8 rows 17.4 us a call, 20.2
// evict-first; 1024 x 64000 26.2, 24.7.  A template parameter: a branch between
// the two forms in the producer's loop cost steps of two row tiles 4 %, a policy
// operand with the normal priority small weights 5 % and steps of three row
// tiles and more, which read W mostly from L2, 1.5 %.
__host__ inline bool pair_w_first(int V, int H, bool in_place) {
  return 2ll * V * H > (in_place ? 115ll : 95ll) << 20;
}

__host__ __device__ inline size_t pair_smem_bytes(int n_stages, bool swap) {
  return 1024 + static_cast<size_t>(n_stages) * kPairStageBytes + (swap ? kSwapXchBytes : 0) +
         static_cast<size_t>(2 * kPairMaxRing + 9) * 8 + 16 + 3 * kPairHalf * 4;
}

// For the pair kernel: blocks of `run` rows x 64 columns, the K blocks of a run
// one after the other, rows >= V of the last run zero.  The kernel reads it
// through a tensor map of 64 columns with no swizzle: K block kb of row r (r /
// run = q) is map row q run KB + kb run + r - q run.  Two runs are used
// (pair_w_run):
//   128, when every tile is 128 rows high: a tile's K blocks are contiguous;
//   all round8(V) rows, otherwise: any run of 8-row atoms of a K block is one
//   contiguous block, so steps of one row tile may cut V evenly (pair_even_rows)
//   and wider ones in 128-row tiles.  Reading 128-row tiles in this order is
//   0.6 % slower (152064 x 3584, M = 96: 169.2 us a step against 170.5).
__global__ void pack_w_tiles_kernel(const uint4* __restrict__ W, uint4* __restrict__ out, int V,
                                    int H, int run, int units,
                                    const __nv_bfloat16* __restrict__ gw) {
  const long long KB = H / kPairBlockK;
  pack_units(W, out, V, H, units, gw, [=](int u) {
    const long long row = static_cast<long long>(u) * kUnitRows;
    const long long q = row / run;
    return PackDst{(q * run * KB + row - q * run) * 128, run * 128ll};
  });
}

// Rows per run of the packed W, and its rows of 64 columns.
__host__ __device__ inline int pair_w_run(int V, int th1) {
  return th1 == kPairHalf ? kPairHalf : (V + 7) / 8 * 8;
}
__host__ __device__ inline long long pair_w_rows(int V, int H, int run) {
  return static_cast<long long>((V + run - 1) / run) * run * (H / kPairBlockK);
}

struct PairSmem {
  uint8_t* stage;      // n_stages x kPairStageBytes: the ring (A half, B half per stage)
  float4* xch;         // swapped orientation: 2 x [4 quarters][256 columns] triples
  uint64_t* full;      // kPairMaxRing (even CTA): both CTAs' halves of the stage landed
  uint64_t* empty;     // kPairMaxRing: the pair's MMAs are done with the stage
  uint64_t* accf;      // 2: accumulator ready
  uint64_t* acce;      // 2 (even CTA): accumulator drained by both epilogues
  uint64_t* drain;     // 1 (even CTA): abort path, issued MMAs complete
  uint64_t* xchb;      // 2 (swapped): the epilogue warps wrote xch[buffer]
  uint64_t* xcub;      // 2 (unswapped): the odd half's warps wrote xchu, the even half's read it
  float* xchu;         // unswapped orientation: [3][128] triples of the odd half
  uint32_t* tmem_slot;
  volatile int* abort;
};

__device__ __forceinline__ PairSmem pair_carve(uint8_t* raw, int n_stages, bool swap) {
  PairSmem s;
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  s.stage = base;
  uint8_t* after = base + static_cast<size_t>(n_stages) * kPairStageBytes;
  s.xch = reinterpret_cast<float4*>(after);
  if (swap) after += kSwapXchBytes;
  s.full = reinterpret_cast<uint64_t*>(after);
  s.empty = s.full + kPairMaxRing;
  s.accf = s.empty + kPairMaxRing;
  s.acce = s.accf + 2;
  s.drain = s.acce + 2;
  s.xchb = s.drain + 1;
  s.xcub = s.xchb + 2;
  s.tmem_slot = reinterpret_cast<uint32_t*>(s.xcub + 2);
  s.abort = reinterpret_cast<volatile int*>(s.tmem_slot + 1);
  s.xchu = reinterpret_cast<float*>(s.tmem_slot + 4);
  return s;
}

struct PairRing {
  int slot = 0;
  uint32_t phase = 0;
  __device__ void next(int n) {
    if (++slot == n) {
      slot = 0;
      phase ^= 1u;
    }
  }
};

__device__ __forceinline__ void pair_drain(uint64_t* bar, uint32_t parity, uint32_t* err) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > kWaitLimitNs) {
      atomicOr(err, kErrDrain);
      return;
    }
  }
}

// kNorm: as in lm_head_softmax_kernel, row n's logits are scaled by inv_r[n]
// (written by the gather).  Swapped steps (pair_swapped) load a tile's rows
// through hm instead of tm_a.
// kStatic: M_fixed rows that the caller passes, known at launch (M <= 256, W
// row-major through the map's own swizzle); the set-up then comes before the
// dependency wait.
template <bool kNorm, bool kStatic, bool kFirst>
__global__ void __cluster_dims__(2, 1, 1) __maxnreg__(kPairRegs)
    lm_head_pair_kernel(const __grid_constant__ CUtensorMap tm_a,
                        const __grid_constant__ CUtensorMap tm_w,
                        const __grid_constant__ CUtensorMap tm_w1,
                        const __grid_constant__ PairRowMaps hm, const PairParams p) {
  extern __shared__ uint8_t smem_raw[];
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();  // 0: even CTA (issues the MMAs), 1: odd
  const int pair = blockIdx.x >> 1;
  const int n_pairs = gridDim.x >> 1;

  // Set-up that does not depend on M, before the dependency wait.
  PairSmem sm = pair_carve(smem_raw, p.n_stages, p.swap_max_n > 0);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kPairMaxRing; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&sm.accf[a], 1);
      mbar_init(&sm.acce[a], 2 * kPairEpiWarps);  // the epilogue warps of both CTAs
      mbar_init(&sm.xchb[a], kPairEpiWarps);      // the epilogue warps of this CTA
      mbar_init(&sm.xcub[a], kPairEpiWarps / 2);  // ... of one half of the columns
    }
    mbar_init(sm.drain, 1);
    *sm.abort = 0;
    fence_mbar_init();
    prefetch_tmap(&tm_a);
    prefetch_tmap(&tm_w);
    prefetch_tmap(&tm_w1);
  }
  if (warp == 1) {
    tmem_alloc_pair(sm.tmem_slot, kPairTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync();  // barriers of both CTAs initialised, tensor memory allocated
  tc_fence_after();
  const uint32_t tmem_base = *sm.tmem_slot;

  int M;
  if constexpr (kStatic) {
    M = p.M_fixed;
    grid_dependency_wait();  // the caller's rows and W, the scratch
    if (blockIdx.x == 0 && threadIdx.x == 0) p.err[1] = 0u;  // the merge's ticket
  } else {
    grid_dependency_wait();  // d_M and the gathered rows of this step
    M = *p.d_M;
  }
  // Every thread (the CTA counts once all of them have), after the wait: the
  // commit kernel, which may start from here, reads the previous step's state
  // before waiting for this kernel.
  grid_launch_dependents();
  if (p.m_hist_slot && blockIdx.x == 0 && threadIdx.x == 0 && (M >= p.min_M || p.min_M <= 1))
    *p.m_hist_slot = M;
  // Nothing to decode here: no tiles, every role falls through.
  const bool none = M < p.min_M || M < 1;
  const bool swap = pair_swapped(M, p.swap_max_n);  // the same in every CTA

  const int KB = p.H / kPairBlockK;
  const int n_rt = none ? 1 : pair_row_tiles(M);
  // Rows per row tile: 256 (the MMA M of the pair), or N when swapped.
  const int rt_rows = swap ? swap_tile_cols(M, n_rt) : kPairTileRows;
  // Vocabulary rows per CTA and tile (half: MMA columns per CTA when unswapped).
  const int th = n_rt == 1 ? p.th1 : kPairHalf;
  const int half = (th + 31) & ~31;
  const int n_tiles = none ? 0 : n_rt == 1 ? p.n_vt1 : p.n_vt * n_rt;
  const int my_tiles = pair < n_tiles ? (n_tiles - pair + n_pairs - 1) / n_pairs : 0;
  // Swapped stages hold the W half and one box of rows_tile / 2 rows, so the
  // ring (n_stages slots of kPairStageBytes) is re-cut to that size: more
  // stages in flight for narrower tiles.  Unswapped steps do not use the
  // swapped epilogue's exchange buffer, which follows the ring: one more stage.
  // K blocks per stage.  Two halve the waits and commits, which bounds narrow
  // tiles of weights that come from L2; only the allocation-free head has them:
  // it also runs blocks of up to 128 rows on this kernel (1088 x 31560, 32 rows
  // 13.5 -> 11.8 us a call, 4096 x 126464 153.0 -> 150.3), while in a context the
  // longer loop cost steps of two row tiles 1.6 %.
  const int kps = kStatic && swap && rt_rows <= kSwapTwoBlocks ? 2 : 1;
  const int rows_bytes = (swap ? rt_rows / 2 : kPairHalf) * kPairBlockK * 2;
  const int stage_stride = kps * (kPairHalfBytes + rows_bytes);
  const int ring_bytes =
      p.n_stages * kPairStageBytes + (!swap && p.swap_max_n > 0 ? kSwapXchBytes : 0);
  const int n_ring = min(p.ring_max, ring_bytes / stage_stride);

  if (warp == 0) {
    // -------------------------------------------------------- producer --
    const uint64_t pol_a = policy_evict_last();
    const uint64_t pol_w = policy_evict_first();
    const uint32_t full0 = mapa_shared(sm.full, 0);  // the even CTA's barriers
    const bool leader = elect_one();
    PairRing r;
    long long issued = 0;
    bool ok = true;
    // Swapped: a CTA's rt_rows / 2 rows (a multiple of 16) load as one box.
    const int q1 = rt_rows / 32 - 1;
    const int box_rows = rt_rows / 2;
    // Bytes of one stage, both CTAs (the even CTA arms its barrier for them).
    const uint32_t stage_tx =
        2u * static_cast<uint32_t>((th + (swap ? box_rows : kPairHalf)) * kPairBlockK * 2);
    const CUtensorMap* tmw = n_rt == 1 ? &tm_w1 : &tm_w;
    for (int i = 0; i < my_tiles && ok; ++i) {
      const int t = pair + i * n_pairs;
      const int v = t / n_rt, j = t - v * n_rt;
      // First row of this CTA's half of the tile's rows.
      const int a_row = j * rt_rows + static_cast<int>(rank) * (swap ? rt_rows / 2 : kPairHalf);
      const int w_row = (2 * v + static_cast<int>(rank)) * th;
      auto load_w = [&](uint8_t* to, uint32_t bar, int kb) {  // K block kb of the W half
        const int x = kb * p.w_dx, y = w_row * p.w_ry + kb * p.w_dy;
        if constexpr (kFirst)
          tma_load_2d_pair(to, tmw, bar, x, y, pol_w);
        else
          tma_load_2d_pair_nohint(to, tmw, bar, x, y);
      };
      for (int kb = 0; kb < KB; kb += kps) {
        ok = ok && mbar_wait(&sm.empty[r.slot], r.phase ^ 1u, sm.abort, p.err, kErrWaitEmpty);
        if (leader && ok) {
          uint8_t* dst = sm.stage + static_cast<size_t>(r.slot) * stage_stride;
          const uint32_t bar = full0 + static_cast<uint32_t>(r.slot * 8);
          // The even CTA arms the stage for the bytes of both CTAs; a copy of
          // the odd CTA that completes first leaves the phase open until then.
          const bool two = kb + 1 < KB && kps > 1;
          if (rank == 0) mbar_arrive_expect_tx(&sm.full[r.slot], two ? 2 * stage_tx : stage_tx);
          if (swap) {
            // A: the W half; B: the CTA's rows, one box of box_rows.  (Two K
            // blocks: W, W, rows, rows.)
            uint8_t* rows = dst + kps * kPairHalfBytes;
            load_w(dst, bar, kb);
            if (two) load_w(dst + kPairHalfBytes, bar, kb + 1);
            tma_load_2d_pair(rows, &hm.box[q1], bar, kb * kPairBlockK, a_row, pol_a);
            if (two)
              tma_load_2d_pair(rows + rows_bytes, &hm.box[q1], bar, (kb + 1) * kPairBlockK, a_row,
                               pol_a);
          } else {
            tma_load_2d_pair(dst, &tm_a, bar, kb * kPairBlockK, a_row, pol_a);
            load_w(dst + kPairHalfBytes, bar, kb);
          }
        }
        __syncwarp();
        issued += ok ? 1 : 0;
        r.next(n_ring);
      }
      ok = __all_sync(0xffffffffu, ok);
    }
    if (!ok && rank == 0 && leader) {
      const long long f0 = issued > n_ring ? issued - n_ring : 0;
      for (long long q = f0; q < issued; ++q)
        pair_drain(&sm.full[q % n_ring], static_cast<uint32_t>((q / n_ring) & 1), p.err);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (rank == 0) {
      // -------------------------------------------- MMA issuer (even CTA) --
      // Swapped: M = 256 vocabulary rows, N = the tile's rows; else M = 256
      // rows, N = 2 half vocabulary rows.
      const uint32_t idesc = idesc_bf16_f32(256, static_cast<uint32_t>(swap ? rt_rows : 2 * half));
      const bool leader = elect_one();
      const uint64_t desc0 = sdesc_k_sw128(smem_addr(sm.stage));
      PairRing r;
      bool ok = true;
      for (int i = 0; i < my_tiles && ok; ++i) {
        const int acc = i & 1;
        ok = __all_sync(0xffffffffu, mbar_wait_cluster(&sm.acce[acc], ((i >> 1) & 1) ^ 1u, sm.abort,
                                                       p.err, kErrWaitAccEmpty));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc * kPairTileVocab);
        for (int kb = 0; kb < KB; kb += kps) {
          ok = ok && mbar_wait_cluster(&sm.full[r.slot], r.phase, sm.abort, p.err, kErrWaitFull);
          tc_fence_after();
          const uint64_t a = desc0 + static_cast<uint32_t>(r.slot * stage_stride >> 4);
          const uint64_t b = a + static_cast<uint32_t>(kps * kPairHalfBytes >> 4);
          if (leader && ok) {
#pragma unroll
            for (int kk = 0; kk < kPairBlockK / 16; ++kk)
              mma_bf16_pair(d_tmem, a + 2 * kk, b + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
            if (kb + 1 < KB && kps > 1) {
              const uint64_t a1 = a + (kPairHalfBytes >> 4);
              const uint64_t b1 = b + static_cast<uint32_t>(rows_bytes >> 4);
#pragma unroll
              for (int kk = 0; kk < kPairBlockK / 16; ++kk)
                mma_bf16_pair(d_tmem, a1 + 2 * kk, b1 + 2 * kk, idesc, 1u);
            }
            mma_commit_pair(&sm.empty[r.slot], 0x3);
          }
          __syncwarp();
          r.next(n_ring);
        }
        ok = __all_sync(0xffffffffu, ok);
        if (leader && ok) mma_commit_pair(&sm.accf[acc], 0x3);
        __syncwarp();
      }
      if (!ok && leader) {
        // Abort: wait for the MMAs already issued (they read both CTAs'
        // shared memory) before anything is released.
        mma_commit_pair(sm.drain, 0x1);
        pair_drain(sm.drain, 0, p.err);
      }
    }
    __syncwarp();
  } else if (swap) {
    // ----------------------------------------------- epilogue (swapped) --
    // The CTA's 128 accumulator lanes are vocabulary rows, its rt_rows columns
    // the tile's rows.  A warp holds 32 lanes and half of the columns, 16 at a
    // time: with 16x256b loads thread (g = lane / 4, h = lane % 4) gets the
    // four lanes g, g + 8, g + 16, g + 24 of the columns 8 j + 2 h + e, and
    // folds them into a running triple per column over all of the pair's
    // tiles.  Only at the end are the eight threads of a column merged
    // (transposing butterfly) and the four warps of a column (through xch).
    const int quarter = warp & 3;  // tensor-memory lanes 32 quarter .. 32 quarter + 31
    const int et = threadIdx.x - 64;
    const int col_half = ((warp - 2) >> 2) * (rt_rows / 2);
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    const uint32_t acce_remote = mapa_shared(sm.acce, 0);
    const int per_row = pair_partials_per_row(M, n_pairs, true);  // > 0: two partials per pair
    const int nch = rt_rows / 32;  // 16-column chunks of this warp
    const int g = lane >> 2, h2 = 2 * (lane & 3);
    float am[4 * kSwapChunks], as[4 * kSwapChunks];
    int aix[4 * kSwapChunks];
    for (int i = 0; i < my_tiles; ++i) {
      const int t = pair + i * n_pairs;
      const int v = t / n_rt, j = t - v * n_rt;
      const int row0 = j * rt_rows;
      const int acc = i & 1;
      // This thread's vocabulary rows; those past the tile (stale stage bytes)
      // or past V count as -inf.
      const int vbase = (2 * v + static_cast<int>(rank)) * th;
      const int vrow = vbase + quarter * 32 + g;
      const int nrow = min(vbase + th, p.V) - vrow;  // rows 8 k < nrow exist
      const bool whole = nrow > 24;
      if (i == 0 || per_row == 0) {
#pragma unroll
        for (int k = 0; k < 4 * kSwapChunks; ++k) {
          am[k] = kNegBig;
          as[k] = 0.0f;
          aix[k] = INT_MAX;
        }
      }
      if (!mbar_wait(&sm.accf[acc], (i >> 1) & 1, sm.abort, p.err, kErrWaitAccFull)) break;
      tc_fence_after();
      const uint32_t tbase = tmem_base + lane_base +
                             static_cast<uint32_t>(acc * kPairTileVocab + col_half);
      uint32_t xa[16], xb[16];
      tmem_ld_16cols_frag(tbase, xa);
#pragma unroll
      for (int c = 0; c < kSwapChunks; ++c) {
        if (c < nch) {
          uint32_t(&x)[16] = (c & 1) ? xb : xa;
          tmem_ld_wait16(x);
          if (c + 1 < kSwapChunks && c + 1 < nch)
            tmem_ld_16cols_frag(tbase + static_cast<uint32_t>(16 * (c + 1)), (c & 1) ? xa : xb);
#pragma unroll
          for (int q = 0; q < 4; ++q) {  // column 8 (q / 2) + h2 + q % 2 of the chunk
            float sc = kLog2e;
            if constexpr (kNorm) {
              const int row = row0 + col_half + 16 * c + 8 * (q >> 1) + h2 + (q & 1);
              if (row < M) sc = kLog2e * __ldg(p.inv_r + row);
            }
            float z[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
              z[k] = __fmul_rn(__uint_as_float(x[8 * (k >> 1) + 4 * (q >> 1) + 2 * (k & 1) + (q & 1)]),
                               sc);
            if (!whole) {
#pragma unroll
              for (int k = 0; k < 4; ++k) z[k] = 8 * k < nrow ? z[k] : -INFINITY;
            }
            fold4(am[4 * c + q], as[4 * c + q], aix[4 * c + q], z, vrow);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (rank == 0)
          mbar_arrive(&sm.acce[acc]);
        else
          mbar_arrive_cluster(acce_remote + static_cast<uint32_t>(acc * 8));
      }
      if (per_row > 0 && i + 1 < my_tiles) continue;
      // One partial per column, of this tile (buffer i & 1 is written again at
      // tile i + 2, after every warp has arrived for tile i + 1, which each
      // does after reading tile i) or, with per_row > 0, of all tiles.
      const int buf = per_row > 0 ? 0 : i & 1;
      float4* xch = sm.xch + buf * 4 * kPairTileVocab + quarter * kPairTileVocab + col_half;
#pragma unroll
      for (int c = 0; c < kSwapChunks; ++c) {
        if (c < nch) {
          float4 f;
          merge_frag8(am + 4 * c, as + 4 * c, aix + 4 * c, lane, f);
          if ((lane & 4) == 0)
            xch[16 * c + ((lane & 16) ? 8 : 0) + h2 + ((lane & 8) ? 1 : 0)] = f;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.xchb[buf]);
      if (!mbar_wait(&sm.xchb[buf], per_row > 0 ? 0u : (i >> 1) & 1, sm.abort, p.err, kErrWaitEpi))
        break;
      if (et < rt_rows && row0 + et < M) {
        float m = kNegBig, sum = 0.0f;
        int ix = INT_MAX;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          const float4 a = sm.xch[(buf * 4 + w) * kPairTileVocab + et];
          merge_tri(m, sum, ix, a.x, a.y, __float_as_int(a.z));
        }
        const size_t row = static_cast<size_t>(row0 + et);
        if (per_row > 0)
          p.part[row * per_row + 2 * (pair / n_rt) + static_cast<int>(rank)] =
              make_float4(m, sum, __int_as_float(ix), 0.0f);
        else if (CAI_IN_RANGE(v < p.n_vt, p.err))
          p.part[row * (2 * p.n_vt) + 2 * v + static_cast<int>(rank)] =
              make_float4(m, sum, __int_as_float(ix), 0.0f);
      }
    }
    if (per_row > 0 && my_tiles == 0 && !none) {
      // A pair without tiles writes the empty triple for its row tile.
      const int row = (pair % n_rt) * rt_rows + et;
      if (et < rt_rows && row < M)
        p.part[static_cast<size_t>(row) * per_row + 2 * (pair / n_rt) + static_cast<int>(rank)] =
            make_float4(kNegBig, 0.0f, __int_as_float(INT_MAX), 0.0f);
    }
  } else {
    // --------------------------------------------------------- epilogue --
    // A tensor-memory lane holds one row's logits; the two warps of a quarter
    // take half of the columns each (the even and the odd CTA's vocabulary
    // rows) and merge their triples through xch.
    const int quarter = warp & 3;  // tensor-memory lanes 32 quarter .. 32 quarter + 31
    const int odd = (warp - 2) >> 2;
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    const uint32_t acce_remote = mapa_shared(sm.acce, 0);
    const int per_row = pair_partials_per_row(M, n_pairs, false);  // > 0: one partial per pair
    float* xm = sm.xchu + quarter * 32 + lane;  // [3][128]: max, sum, index
    float m = kNegBig, s = 0.0f;
    int ix = INT_MAX;
    for (int i = 0; i < my_tiles; ++i) {
      const int t = pair + i * n_pairs;
      const int v = t / n_rt, j = t - v * n_rt;
      const int acc = i & 1;
      if (per_row == 0) {
        m = kNegBig;
        s = 0.0f;
        ix = INT_MAX;
      }
      if (!mbar_wait(&sm.accf[acc], (i >> 1) & 1, sm.abort, p.err, kErrWaitAccFull)) break;
      tc_fence_after();
      const uint32_t tbase = tmem_base + lane_base +
                             static_cast<uint32_t>(acc * kPairTileVocab + odd * half);
      const int row = j * kPairTileRows + static_cast<int>(rank) * kPairHalf + quarter * 32 + lane;
      float rs = kLog2e;
      if constexpr (kNorm) {
        if (row < M) rs = kLog2e * __ldg(p.inv_r + row);
      }
      // Columns [0, half) are the even CTA's th vocabulary rows, [half, 2 half)
      // the odd one's; columns past th (stale stage bytes) or past V are left out.
      const int vbase = (2 * v + odd) * th;
      const int nrow = min(th, p.V - vbase);
#pragma unroll 1
      for (int c = 0; c < half / 32; ++c) {
        uint32_t x[32];
        tmem_ld_32cols(tbase + static_cast<uint32_t>(32 * c), x);
        tmem_ld_wait();
        fold_row32(m, s, ix, x, rs, vbase + 32 * c, nrow - 32 * c);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (rank == 0)
          mbar_arrive(&sm.acce[acc]);
        else
          mbar_arrive_cluster(acce_remote + static_cast<uint32_t>(acc * 8));
      }
      if (per_row > 0 && i + 1 < my_tiles) continue;
      // n-th exchange of this step: the odd half's warps write it once the
      // even half's have read the one before (xcub[1]), and announce it (xcub[0]).
      const int n = per_row > 0 ? 0 : i;
      if (odd) {
        if (n > 0 && !mbar_wait(&sm.xcub[1], (n - 1) & 1, sm.abort, p.err, kErrWaitEpi)) break;
        xm[0] = m;
        xm[kPairHalf] = s;
        xm[2 * kPairHalf] = __int_as_float(ix);
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.xcub[0]);
        continue;
      }
      if (!mbar_wait(&sm.xcub[0], n & 1, sm.abort, p.err, kErrWaitEpi)) break;
      const float om = xm[0], os = xm[kPairHalf];
      const int oix = __float_as_int(xm[2 * kPairHalf]);
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.xcub[1]);
      merge_tri(m, s, ix, om, os, oix);
      if (row < M) {
        if (per_row > 0)
          p.part[static_cast<size_t>(row) * per_row + pair / n_rt] =
              make_float4(m, s, __int_as_float(ix), 0.0f);
        else if (CAI_IN_RANGE(v < p.n_vt, p.err))
          p.part[static_cast<size_t>(row) * p.n_vt + v] =
              make_float4(m, s, __int_as_float(ix), 0.0f);
      }
    }
    if (per_row > 0 && my_tiles == 0 && !none && !odd) {
      // A pair without tiles writes the empty triple for its row tile.
      const int row = (pair % n_rt) * kPairTileRows + static_cast<int>(rank) * kPairHalf +
                      quarter * 32 + lane;
      if (row < M)
        p.part[static_cast<size_t>(row) * per_row + pair / n_rt] =
            make_float4(kNegBig, 0.0f, __int_as_float(INT_MAX), 0.0f);
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();  // no CTA leaves while the pair's MMAs or arrivals may touch it
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, kPairTmemCols);
  }
}

// Second stage of a pair step: one warp per masked row merges the row's
// n_vt tile partials (merge_tri: max, rescaled sum, lowest index among equal
// maxima) into one triple, rowres[row], so that the commit reads one value per
// row.  Returns at once when the step ran on the swapped-operand kernel.
struct ReduceParams {
  const float4* part;  // [rows, n_vt] partials (unswapped step), [rows, 2 n_vt] (swapped)
  float4* rowres;      // [rows]
  const int* d_M;
  int n_vt;
  int min_M;
  int n_pairs;         // the pair kernel's grid / 2 (its partials need no merge when
                       // pair_partials_per_row > 0)
  int swap_max_n;      // the pair kernel's orientation rule (pair_swapped)
};

constexpr int kReduceThreads = 256;

__global__ void __launch_bounds__(kReduceThreads) reduce_partials_kernel(const ReduceParams p) {
  grid_launch_dependents();  // every thread: the CTA counts once all of them have
  grid_dependency_wait();    // the pair kernel's partials
  const int M = *p.d_M;
  const bool swap = pair_swapped(M, p.swap_max_n);
  if (M < p.min_M || M < 1 || pair_partials_per_row(M, p.n_pairs, swap) > 0) return;
  const int n_part = (swap ? 2 : 1) * p.n_vt;
  const int lane = threadIdx.x & 31;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < M; row += nw) {
    const float4* pr = p.part + static_cast<size_t>(row) * n_part;
    float m = kNegBig, s = 0.0f;
    int ix = INT_MAX;
    int k = lane;
    for (; k + 96 < n_part; k += 128) {  // four loads in flight per lane
      const float4 a = __ldcg(pr + k), b = __ldcg(pr + k + 32), c = __ldcg(pr + k + 64),
                   d = __ldcg(pr + k + 96);
      merge_tri(m, s, ix, a.x, a.y, __float_as_int(a.z));
      merge_tri(m, s, ix, b.x, b.y, __float_as_int(b.z));
      merge_tri(m, s, ix, c.x, c.y, __float_as_int(c.z));
      merge_tri(m, s, ix, d.x, d.y, __float_as_int(d.z));
    }
    for (; k < n_part; k += 32) {
      const float4 a = __ldcg(pr + k);
      merge_tri(m, s, ix, a.x, a.y, __float_as_int(a.z));
    }
    __syncwarp();
    const float4 q[1] = {make_float4(m, s, __int_as_float(ix), 0.0f)};
    warp_merge(q, m, s, ix);
    if (lane == 0) p.rowres[row] = make_float4(m, s, __int_as_float(ix), 0.0f);
  }
}

}  // namespace cai
