// LM head of the single-kernel step with the masked rows as the MMA's A
// operand: the same quantities as lm_head_softmax_kernel (Box 1 of
// arXiv 2608.22646: c_i = max_v p_theta(x_i = v) and argmax_v p_theta,
// logits never leaving tensor memory), for the M <= 128 rows of a step whose
// block holds at most 128 positions.
//
// Why this orientation.  In the swapped kernel (lm_head_softmax_kernel, W as
// the A operand, the rows as N = 32) every 16 KiB W stage took ~0.345 us of
// the MMA thread (four K = 16 MMAs, their waits and commits), whatever the
// stage held: ~48 GB/s of W per SM, the HBM share of 151 SMs, so the stream
// was paced by the MMA side and a CTA's short last tile cost as much as a
// full one (the same stream without MMAs, or with one MMA per stage, ran at
// 7.7-7.8 TB/s).  With the rows as A and up to 256 vocabulary rows as B, a
// 32 KiB stage of W takes four MMAs, half as many per byte, and the stream is
// HBM-bound.  The rows pad to M = 128, which the tensor cores absorb (an
// M = 128, N = 256, K = 16 MMA takes ~65 ns on resident operands).
//
// Rows stages.  The MMA reads 128 rows of A, but only the first mq =
// round16(M) are the step's; the accumulator rows past M are never read.  So
// the rows part of a K block owns only mq rows (the parts lie mq * 128 bytes
// rounded up to 1 KiB apart, 4 KiB for M <= 32, before the W parts) and the
// MMA's read of the other rows runs on into the following parts (and, for the
// last ones, the W ring): whatever it finds there only reaches accumulator rows
// that no thread loads.  A stage's rows and W complete one barrier and are
// freed by one commit; with a ring and barriers of their own for the rows a
// stage took two waits and two commits: 1024 x 22000 11.3 us a step, now 10.0;
// 2048 x 50003 30.0, now 27.1; 4096 x 126464 with 128 rows 141.8, now 134.2
// (the figures of this file at 65 to 128 rows: steps back to back without the
// wait for their rows, HeadParams::wait_rows, which adds 4 to 12 us to each).
//
// Work split: as lm_head_softmax_kernel, V in units of 8 rows over the CTAs;
// a CTA's rows form equal groups of at most 256 vocabulary rows (RowsPlan),
// and the packed W (pack_weight_rows_kernel) stores each group's K block as
// one contiguous block of at most 32 KiB in the 128-byte-swizzled K-major
// layout, so one bulk copy loads one B stage.  The
// CTA runs its groups one after the other, each over all K blocks into one of
// two tensor-memory accumulators (128 lanes x 256 columns); the rows' K block
// is reloaded (from L2) for every group, as one box of round16(M) rows.
//
// The producer and the MMA warp run their loops with all lanes and issue from
// one (see the pair kernel): alone, LLaDA's 32 rows 160.6 -> 159.6 us and 64
// rows 168.4 -> 166.6 us; back to back 1.5 % of a generation.
//
// Roles (320 threads): warp 0 producer (W stages by bulk copy, row stages by
// TMA); warp 1 allocates tensor memory and issues the MMAs; warps 2..9
// epilogue: tensor-memory lane r holds row r's logits, so
// two threads (half of the columns each) run a serial online softmax over the
// group's columns (only warps whose 32 lanes hold rows < M have work).  One of
// them writes one partial per (row, CTA); the last CTA merges them and commits the step
// (fused_step_commit), as in the single-kernel step of
// lm_head_softmax_kernel, with the same cross-step behaviour under
// programmatic dependent launch.
#pragma once

#include <climits>
#include "head_kernel.cuh"
#include "ptx.cuh"
#include "softmax.cuh"

namespace cai {

constexpr int kRowsM = 128;                          // MMA M: rows of the step, padded
constexpr int kRowsGroupRows = 256;                  // MMA N: vocabulary rows per group
constexpr int kRowsTmemCols = 2 * kRowsGroupRows;    // two accumulators
constexpr int kRowsEpiWarps = 8;                     // two per tensor-memory quarter
constexpr int kRowsThreads = 64 + 32 * kRowsEpiWarps;

// Bytes between two rows stages for a step of M rows (see above).
__host__ __device__ inline int rows_h_stride(int M) {
  return (((M + 15) & ~15) * 128 + 1023) & ~1023;
}

// The rows ring comes first, then the W ring, whose first 12 KiB or more
// cover the last rows stage's read past its own bytes.
__host__ __device__ inline size_t rows_smem_bytes(int n_stages, int w_stage, int h_stage) {
  return 1024 + static_cast<size_t>(n_stages) * (h_stage + w_stage) +
         static_cast<size_t>(2 * n_stages + 6) * 8 + 16;
}

struct RowsSmem {
  uint8_t* h;         // n_stages x h_stride
  uint8_t* w;         // n_stages x w_stage
  uint64_t* full;     // n_stages: the stage's W and rows landed
  uint64_t* empty;    // n_stages: the MMAs are done with the stage
  uint64_t* accf;     // 2: accumulator ready
  uint64_t* acce;     // 2: accumulator drained by the epilogue warps
  uint64_t* drain;    // 1
  uint64_t* xch;      // 1: the second half's epilogue warps wrote their triples
  uint32_t* tmem_slot;
  volatile int* abort;
  volatile int* skip;
};

__device__ __forceinline__ RowsSmem rows_carve(uint8_t* raw, int n_stages, int w_stage,
                                               int h_stage) {
  RowsSmem s;
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  s.h = base;
  s.w = s.h + static_cast<size_t>(n_stages) * h_stage;
  s.full = reinterpret_cast<uint64_t*>(s.w + static_cast<size_t>(n_stages) * w_stage);
  s.empty = s.full + n_stages;
  s.accf = s.empty + n_stages;
  s.acce = s.accf + 2;
  s.drain = s.acce + 2;
  s.xch = s.drain + 1;
  s.tmem_slot = reinterpret_cast<uint32_t*>(s.xch + 1);
  s.abort = reinterpret_cast<volatile int*>(s.tmem_slot + 1);
  s.skip = s.abort + 1;
  return s;
}

// The work of one CTA: units [u0, u1) of kUnitRows rows (the same split of V
// as lm_head_softmax_kernel), cut into n_groups = ceil(rows / 256) groups of
// equal size to within one unit.  Equal groups keep every group's MMAs (whose
// time hardly depends on N) under its share of the W stream; a short last
// group would be paced by its MMAs instead.
struct RowsPlan {
  int u0, u1, n_groups;
  __host__ __device__ int row0() const { return u0 * kUnitRows; }
  __host__ __device__ int rows() const { return (u1 - u0) * kUnitRows; }
  // First unit of group g, relative to u0.
  __host__ __device__ int group_unit(int g) const {
    return static_cast<int>((static_cast<long long>(g) * (u1 - u0)) / n_groups);
  }
  __host__ __device__ int group_row0(int g) const { return row0() + group_unit(g) * kUnitRows; }
  __host__ __device__ int group_rows(int g) const {
    return (group_unit(g + 1) - group_unit(g)) * kUnitRows;
  }
  // Byte offset in the packed weight of group g's K block kb: a group's K
  // blocks follow one another, each group_rows(g) x 128 bytes.
  __host__ __device__ size_t stage_offset(int g, int kb, int H) const {
    return static_cast<size_t>(group_row0(g)) * 2 * H +
           static_cast<size_t>(kb) * group_rows(g) * 128;
  }
};

// W stages of one K block: at least four, and with a long K five while about
// 128 KiB of weight are in flight per SM.  Deeper rings stream faster on most SMs but starve some (LLaDA
// shape: finish spread 4 us at four 27 KiB stages, 20 us at six), and a step
// waits for its slowest CTA; a short K pays for filling a deeper ring (1024 x
// 40000: 17.3 us a step at four stages, 18.3 at eight; 3584 x 80000: 77.1 at
// four, 75.0 at five, 75.1 at eight).
constexpr int kRowsInFlight = 128 << 10;

// K blocks per stage, given the bytes of one block's W and rows parts: two
// where four such stages fit, or three and the weight stays in L2.  A stage's
// waits, commit and copies take ~0.25 us whatever it holds, which bounds
// weights that come from L2 (1024 x 10000 9.0 -> 7.8 us a step, 1024 x 40000 15.4
// -> 13.3, 2048 x 50003 27.4 -> 24.6).  At the memory's rate it makes no
// difference back to back, but three stages of 64 KiB start a lone step later
// (3584 x 152064 161.8 -> 164.6 us), and with two in flight the stream stalls
// (4096 x 126464, 128 rows: 136.4 -> 143).
__host__ inline int rows_k_blocks(int V, int H, int w_bytes, int h_bytes, size_t smem_limit) {
  const int need = 2ll * V * H <= 128ll << 20 ? 3 : 4;
  return H >= 2 * kBlockK && rows_smem_bytes(need, 2 * w_bytes, 2 * h_bytes) <= smem_limit ? 2 : 1;
}

__host__ __device__ inline RowsPlan rows_plan(int c, int units, int G) {
  RowsPlan p;
  p.u0 = unit_begin(c, units, G);
  p.u1 = unit_begin(c + 1, units, G);
  p.n_groups = (p.rows() + kRowsGroupRows - 1) / kRowsGroupRows;
  return p;
}

// For lm_head_rows_kernel on G CTAs: CTA c's groups in order, each group's K
// blocks in order, each K block the group's rows.
__global__ void pack_weight_rows_kernel(const uint4* __restrict__ W, uint4* __restrict__ out, int V,
                                        int H, int units, int G,
                                        const __nv_bfloat16* __restrict__ gw) {
  pack_units(W, out, V, H, units, gw, [=](int u) {
    const RowsPlan pl = rows_plan(unit_owner(u, units, G), units, G);
    // Group holding unit u (groups are whole units).
    int g = static_cast<int>((static_cast<long long>(u - pl.u0) * pl.n_groups) / (pl.u1 - pl.u0));
    while (g + 1 < pl.n_groups && pl.group_unit(g + 1) <= u - pl.u0) ++g;
    while (g > 0 && pl.group_unit(g) > u - pl.u0) --g;
    return PackDst{static_cast<long long>(pl.stage_offset(g, 0, H)) +
                       (u - pl.u0 - pl.group_unit(g)) * (kUnitRows * 128),
                   static_cast<long long>(pl.group_rows(g)) * 128};
  });
}

// Single-kernel step only (p.fused = 1, p.M_fixed <= 128), W packed by
// pack_weight_rows_kernel.  p.n_stages is the W ring depth (p.w_stage bytes each),
// p.n_bslots the rows ring depth (stages rows_h_stride(M) apart).  kNorm: row
// r's logits are scaled by 1 / sqrt(mean h^2 + eps) of the row, which the
// epilogue warps compute from the step's rows (p.hid).
template <bool kNorm>
__global__ void __launch_bounds__(kRowsThreads, 1)
    lm_head_rows_kernel(const __grid_constant__ CUtensorMap tm_h, const HeadParams p) {
  extern __shared__ uint8_t smem_raw[];
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int h_stride = rows_h_stride(p.M_fixed);
  RowsSmem sm = rows_carve(smem_raw, p.n_stages, p.w_stage, p.kps * h_stride);
  const int cta = blockIdx.x;
  const RowsPlan pl = rows_plan(cta, p.units, gridDim.x);
  const int KB = p.H / kBlockK;
  const int M = p.M_fixed;
  const int mq = (M + 15) & ~15;  // rows loaded per K block (TMA fills rows past B P with zeros)
  const bool spec = !p.first;     // may find out that nothing is masked
  const int n_pre = p.prefetch ? min(p.n_stages, pl.n_groups * ((KB + p.kps - 1) / p.kps)) : 0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.n_stages; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&sm.accf[a], 1);
      mbar_init(&sm.acce[a], kRowsEpiWarps);
    }
    mbar_init(sm.drain, 1);
    mbar_init(sm.xch, kRowsEpiWarps / 2);
    *sm.abort = 0;
    *sm.skip = 0;
    fence_mbar_init();
    // The weight does not depend on earlier kernels: the first ring of W
    // stages is issued now, before the tensor-memory allocation.
    const uint64_t pol_w = policy_evict_first();
    int i = 0;
    for (int g = 0; g < pl.n_groups && i < n_pre; ++g)
      for (int kb = 0; kb < KB && i < n_pre; kb += p.kps, ++i) {
        const uint32_t bytes = static_cast<uint32_t>(pl.group_rows(g) * 128 * min(p.kps, KB - kb));
        mbar_expect_tx(&sm.full[i], bytes);
        bulk_load(sm.w + static_cast<size_t>(i) * p.w_stage,
                  p.wpk + pl.stage_offset(g, kb, p.H), bytes, &sm.full[i], pol_w);
      }
  }
  grid_launch_dependents();  // every thread: the CTA counts once all of them have
  if (warp == 0 && lane == 0) prefetch_tmap(&tm_h);
  if (warp == 1) {
    tmem_alloc(sm.tmem_slot, kRowsTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *sm.tmem_slot;
  // Every role: the bounded waits of one for another must not include the kernel
  // before this one, however long that takes.
  if (p.wait_rows) grid_dependency_wait();

  bool buffers_free = false;  // thread 0: see fused_step_commit
  if (warp == 0) {
    // -------------------------------------------------------- producer --
    // The whole warp runs the loop and one lane issues (see the pair
    // kernel).  A lane whose wait gave up only stops waiting and issuing; the
    // warp leaves together at the end of the group.
    const uint64_t pol_w = policy_evict_first();
    const uint64_t pol_h = policy_evict_last();
    const bool leader = elect_one();
    Ring r;
    int issued = 0;
    bool ok = true, decided = !spec;
    // Rows copied from the host on the context's side stream: wait (bounded)
    // for that copy's sequence word before the first row load.
    if (leader && p.stage_word &&
        !wait_word_ge(p.stage_word, p.stage_seq, sm.abort, p.err, kErrWaitRows))
      ok = false;
    ok = __all_sync(0xffffffffu, ok);
    // The previous step's published word, loaded one K block ahead of its use.
    unsigned long long pub_w = spec ? load_pub(p.cp.pub) : 0ull;
    for (int g = 0; g < pl.n_groups && ok; ++g) {
      const uint32_t wbytes = static_cast<uint32_t>(pl.group_rows(g) * 128);
      const uint8_t* wsrc = p.wpk + pl.stage_offset(g, 0, p.H);
      for (int kb = 0; kb < KB; kb += p.kps) {
        ok = ok && mbar_wait(&sm.empty[r.slot], r.phase ^ 1u, sm.abort, p.err, kErrWaitEmpty);
        if (!decided &&
            previous_left_nothing(__shfl_sync(0xffffffffu, pub_w, 0), p.cp.step_id, decided)) {
          // Stop: the stage completes without rows and carries the stop mark,
          // this K block's number, to the MMA warp, which consumes every
          // stage issued before it first (no copy may be in flight when the
          // CTA leaves or its shared memory is used for the commit).
          if (leader && ok) {
            *sm.skip = g * KB + kb + 1;
            mbar_arrive(&sm.full[r.slot]);
          }
          issued += ok ? 1 : 0;
          g = pl.n_groups;
          break;
        }
        if (!decided) pub_w = load_pub(p.cp.pub);
        if (leader && ok) {
          const bool pre = issued < n_pre;  // the W copy is already in flight
          const uint32_t nk = static_cast<uint32_t>(min(p.kps, KB - kb));
          mbar_arrive_expect_tx(&sm.full[r.slot], nk * (static_cast<uint32_t>(mq * 128) +
                                                        (pre ? 0u : wbytes)));
          uint8_t* h = sm.h + r.slot * p.kps * h_stride;
          tma_load_2d(h, &tm_h, &sm.full[r.slot], kb * kBlockK, 0, pol_h);
          if (nk > 1)
            tma_load_2d(h + h_stride, &tm_h, &sm.full[r.slot], (kb + 1) * kBlockK, 0, pol_h);
          if (!pre)
            bulk_load(sm.w + r.slot * p.w_stage, wsrc + static_cast<size_t>(kb) * wbytes,
                      nk * wbytes, &sm.full[r.slot], pol_w);
        }
        __syncwarp();
        issued += ok ? 1 : 0;
        r.next(p.n_stages);
      }
      ok = __all_sync(0xffffffffu, ok);
    }
    if (leader) {
      if (issued < n_pre) {
        // A stop or an abort before the prefetched stages were claimed:
        // complete their phases so the copies can drain.
        for (int i = issued; i < n_pre; ++i) mbar_arrive(&sm.full[i]);
        for (int i = issued; i < n_pre; ++i) mbar_drain(&sm.full[i], 0, p.err);
      }
      if (!ok) {
        // Abort path: let the copies already in flight land before exit.
        for (int i = issued > p.n_stages ? issued - p.n_stages : 0; i < issued; ++i)
          mbar_drain(&sm.full[i % p.n_stages], static_cast<uint32_t>((i / p.n_stages) & 1), p.err);
      }
    }
    __syncwarp();
    if (lane == 0) buffers_free = step_buffers_free(p.cp, p.first != 0);
  } else if (warp == 1) {
    // ------------------------------------------------------ MMA issuer --
    const bool leader = elect_one();
    const uint64_t h_desc = sdesc_k_sw128(smem_addr(sm.h));
    const uint64_t w_desc = sdesc_k_sw128(smem_addr(sm.w));
    Ring r, racc;
    bool ok = true, skipped = false;
    for (int g = 0; g < pl.n_groups && ok && !skipped; ++g) {
      const uint32_t n = static_cast<uint32_t>((pl.group_rows(g) + 15) & ~15);
      const uint32_t idesc = idesc_bf16_f32(kRowsM, n);
      ok = __all_sync(0xffffffffu, mbar_wait(&sm.acce[racc.slot], racc.phase ^ 1u, sm.abort, p.err,
                                             kErrWaitAccEmpty));
      if (!ok) break;
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(racc.slot * kRowsGroupRows);
      const uint32_t w_next = static_cast<uint32_t>(pl.group_rows(g) * 128) >> 4;
      for (int kb = 0; kb < KB; kb += p.kps) {
        ok = ok && mbar_wait(&sm.full[r.slot], r.phase, sm.abort, p.err, kErrWaitFull);
        if (spec && __any_sync(0xffffffffu, ok && *sm.skip == g * KB + kb + 1)) {
          skipped = true;
          break;
        }
        tc_fence_after();
        const uint64_t a = h_desc + static_cast<uint32_t>(r.slot * p.kps * h_stride >> 4);
        const uint64_t b = w_desc + static_cast<uint32_t>(r.slot * p.w_stage >> 4);
        if (leader && ok) {
#pragma unroll
          for (int kk = 0; kk < kBlockK / 16; ++kk)
            mma_bf16(d_tmem, a + 2 * kk, b + 2 * kk, idesc, (kb | kk) != 0 ? 1u : 0u);
          if (kb + 1 < KB && p.kps > 1) {
            const uint64_t a1 = a + static_cast<uint32_t>(h_stride >> 4), b1 = b + w_next;
#pragma unroll
            for (int kk = 0; kk < kBlockK / 16; ++kk)
              mma_bf16(d_tmem, a1 + 2 * kk, b1 + 2 * kk, idesc, 1u);
          }
          mma_commit(&sm.empty[r.slot]);
        }
        __syncwarp();
        r.next(p.n_stages);
      }
      ok = __all_sync(0xffffffffu, ok);
      if (!ok || skipped) break;
      if (leader) mma_commit(&sm.accf[racc.slot]);
      __syncwarp();
      racc.next(2);
    }
    if (leader) {
      if (!ok || skipped) {
        // Abort or stop: wait for every MMA already issued before tensor
        // memory is freed, then release the epilogue.
        mma_commit(sm.drain);
        mbar_drain(sm.drain, 0, p.err);
      }
      if (skipped) mbar_arrive(&sm.accf[racc.slot]);
    }
    __syncwarp();
  } else {
    // --------------------------------------------------------- epilogue --
    const int quarter = warp & 3;  // tensor-memory lanes 32 quarter .. 32 quarter + 31
    const int hf = (warp - 2) >> 2;  // half of a group's 32-column chunks
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    const int row = quarter * 32 + lane;
    const bool active = quarter * 32 < M;  // warp-uniform: some lane holds a row
    float m = kNegBig, s = 0.0f;
    int ix = INT_MAX;
    float rs = kLog2e;
    if constexpr (kNorm) {
      // The final RMSNorm's row scales, from the step's rows while the first
      // group accumulates.  Nothing here waits for an earlier kernel (with
      // wait_rows every role has, above), so the accumulators are drained as in a step without the norm.
      __shared__ float s_scale[kRowsM];
      epilogue_row_scales<kRowsEpiWarps>(p.hid, M, p.H, p.norm_eps, s_scale, warp - 2, lane);
      if (row < M) rs = kLog2e * s_scale[row];
    }
    Ring racc;
    bool ok = true;
    bool free_now = false;  // looked up early: the load is not waited for at the end
    for (int g = 0; g < pl.n_groups; ++g) {
      if (g == pl.n_groups - 1) free_now = step_buffers_free(p.cp, p.first != 0);
      if (!mbar_wait(&sm.accf[racc.slot], racc.phase, sm.abort, p.err, kErrWaitAccFull)) {
        ok = false;
        break;
      }
      const int stop = spec ? *sm.skip : 0;
      if (stop > g * KB && stop <= (g + 1) * KB) {
        ok = false;  // stopped in this group: nothing of this step is written
        break;
      }
      tc_fence_after();
      if (active) {
        const uint32_t tbase =
            tmem_base + lane_base + static_cast<uint32_t>(racc.slot * kRowsGroupRows);
        const int vbase = pl.group_row0(g);
        // Vocabulary rows past the group's (stale stage bytes) or past V are left out.
        const int nrow = min(pl.group_rows(g), p.V - vbase);
        const int nch = (pl.group_rows(g) + 31) >> 5;
        const int c1 = hf ? nch : (nch + 1) >> 1;
#pragma unroll 1
        for (int c = hf ? (nch + 1) >> 1 : 0; c < c1; ++c) {
          uint32_t x[32];
          tmem_ld_32cols(tbase + static_cast<uint32_t>(32 * c), x);
          tmem_ld_wait();
          fold_row32(m, s, ix, x, rs, vbase + 32 * c, nrow - 32 * c);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.acce[racc.slot]);
      racc.next(2);
    }
    // The second half's triples go through shared memory to the first's.
    __shared__ float s_x[3][kRowsM];
    if (ok && hf) {
      s_x[0][row] = m;
      s_x[1][row] = s;
      s_x[2][row] = __int_as_float(ix);
      __syncwarp();
      if (lane == 0) mbar_arrive(sm.xch);
    } else if (ok && active &&
               mbar_wait(sm.xch, 0, sm.abort, p.err, kErrWaitEpi) && row < M) {
      merge_tri(m, s, ix, s_x[0][row], s_x[1][row], __float_as_int(s_x[2][row]));
      // The step before last read the same partial buffer.
      if (!free_now && !step_buffers_free(p.cp, p.first != 0)) grid_dependency_wait();
      p.part[static_cast<size_t>(row) * gridDim.x + cta] = make_float4(m, s, __int_as_float(ix), 0.0f);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kRowsTmemCols);
  }
  fused_step_commit(p.cp, sm.w, buffers_free);
}

}  // namespace cai
