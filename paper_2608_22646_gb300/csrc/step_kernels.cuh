// The two light kernels around the LM head in one denoising step:
//   gather_rows_kernel    copies the hidden rows of the step's masked
//                         positions into the compact [rows_cap, H] operand;
//   merge_commit_kernel   merges the per-CTA softmax partials into c_i and the
//                         argmax, then runs the commit rule of Algorithm 1
//                         (arXiv 2608.22646) for one sequence per CTA; the last
//                         CTA to finish builds the next step's masked-row list.
#pragma once

#include <cuda_bf16.h>
#include "head_kernel.cuh"
#include "pair_kernel.cuh"

namespace cai {

constexpr int kGatherRowsPerCta = 4;
constexpr int kGatherVecs = 8;       // 16-byte loads in flight per gather thread (H <= 4096 in one round)
constexpr int kGatherThreads = 256;
constexpr int kListThreads = 256;    // rebuild_list_kernel
// Merge kernel: one CTA per sequence, 16 warps of 4 positions each, so that
// a 64-position block merges in one round of loads and the last CTA builds
// the next step's list 512 tokens at a time (measured against 256 threads of
// 6 positions: see the design notes).
constexpr int kCommitThreads = 512;
constexpr int kCommitPPW = 4;

// ------------------------------------------------------------ gather (K1) --

struct GatherParams {
  const __nv_bfloat16* hidden;  // [B P, H] hidden states of the current block
  __nv_bfloat16* hc;            // [rows_cap, H] compact operand of the LM head
  int* list;                    // [B P] token (b P + p) of each masked row
  int* row_of;                  // [B P] row of each token in this step's list, -1
  int* d_M;                     // masked rows of this step
  uint32_t* err;                // error word (CAI_DEBUG range checks)
  int B, BP, H;
  int first;                    // step zero: every position of every sequence
  float* inv_r;                 // final norm: 1 / sqrt(mean h^2 + eps) per row, or null
  float eps;
  const unsigned long long* stage_word;  // host rows staged by the side stream: read
  unsigned long long stage_seq;          // once *stage_word >= stage_seq (or null)
  int prefetch;  // hidden is device memory that holds the rows already
};

__global__ void __launch_bounds__(kGatherThreads)
    gather_rows_kernel(const GatherParams p) {
  grid_launch_dependents();  // every thread: the CTA counts once all of them have
  if (!p.first && p.prefetch) {
    // While the previous step commits: the rows of its list, of which this
    // step's is a part, towards L2 (the weight has passed through it since).
    const int q = blockIdx.x * kGatherRowsPerCta + threadIdx.x / 64;
    const int row = q < p.BP ? __ldcg(p.list + q) : -1;  // stale past the old list
    if (row >= 0 && row < p.BP) {
      const char* src = reinterpret_cast<const char*>(p.hidden) + static_cast<size_t>(row) * p.H * 2;
      for (int o = (threadIdx.x & 63) * 128; o < 2 * p.H; o += 64 * 128) prefetch_l2(src + o);
    }
  }
  grid_dependency_wait();  // the previous step's merge wrote list, row_of and d_M
  if (p.stage_word) {
    // The side stream's copy of the rows: one thread waits (bounded) for its
    // word; on giving up the error word is set and the step's results are
    // not to be used (the host reads the error with them).
    __shared__ volatile int s_abort;
    if (threadIdx.x == 0) {
      s_abort = 0;
      wait_word_ge(p.stage_word, p.stage_seq, &s_abort, p.err, kErrWaitRows);
    }
    __syncthreads();
  }
  // (the row of the list does not wait for M)
  const int r = blockIdx.x * kGatherRowsPerCta + threadIdx.x / 64;
  int src_row = p.first || r >= p.BP ? r : __ldcg(p.list + r);
  const int M = p.first ? p.BP : __ldcg(p.d_M);
  if (p.first) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < p.BP; i += gridDim.x * blockDim.x) {
      p.list[i] = i;
      p.row_of[i] = i;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *p.d_M = p.BP;
  }
  const int rows_pad = (M + 15) & ~15;
  const int t = threadIdx.x & 63;
  const int nvec = p.H / 8;  // 16-byte vectors per row
  float ss = 0.0f;
  if (r < rows_pad) {
    uint4* dst = reinterpret_cast<uint4*>(p.hc + static_cast<size_t>(r) * p.H);
    if (r < M) {
      if (!CAI_IN_RANGE(src_row >= 0 && src_row < p.BP, p.err)) src_row = 0;
      const uint4* src =
          reinterpret_cast<const uint4*>(p.hidden + static_cast<size_t>(src_row) * p.H);
      // All of a thread's loads are issued before its first store (the
      // compiler cannot reorder them: dst and src could alias as far as it
      // knows), so a row costs one memory round trip, not one per vector.
      for (int v0 = t; v0 < nvec; v0 += 64 * kGatherVecs) {
        uint4 x[kGatherVecs];
#pragma unroll
        for (int j = 0; j < kGatherVecs; ++j) {
          const int v = v0 + 64 * j;
          x[j] = v < nvec ? __ldg(src + v) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int j = 0; j < kGatherVecs; ++j) {
          const int v = v0 + 64 * j;
          if (v < nvec) {
            dst[v] = x[j];
            if (p.inv_r) ss += sumsq8(x[j]);
          }
        }
      }
    } else {
      for (int v = t; v < nvec; v += 64) dst[v] = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  if (!p.inv_r) return;
  // A row's 64 threads are two whole warps: reduce in each, then across the two.
  __shared__ float s_half[kGatherThreads / 32];
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
  if ((threadIdx.x & 31) == 0) s_half[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (t == 0 && r < rows_pad) {
    const float tot = s_half[threadIdx.x >> 5] + s_half[(threadIdx.x >> 5) + 1];
    p.inv_r[r] = r < M ? rsqrtf(tot / static_cast<float>(p.H) + p.eps) : 1.0f;
  }
}

// ----------------------------------------------------------- diagnostics --

struct DriftParams {
  const __nv_bfloat16* hidden;  // [B P, H] this step's rows (every position of the block)
  __nv_bfloat16* prev;          // [B P, H] the previous step's rows (kept by this kernel)
  float* ratio;                 // [B P] relative change of each row
  unsigned* count;              // [B] rows of a sequence done, zero between launches
  float* drift;                 // [B, n_blocks, T]
  int BP, P, H, n_blocks, T, blk, t;
};

constexpr int kDriftRowsPerCta = 4;  // one warp per row
constexpr int kDriftVecs = 8;        // 16-byte loads in flight per lane and operand

// One warp per position: ||h^(t) - h^(t-1)|| / ||h^(t-1)|| (Eq. relative_drift;
// fp32 sums of the bf16 rows), then this step's row becomes the previous one
// (at t = 0 only that copy is made).  The warp that finishes a sequence's last
// row averages the P ratios, in a fixed order, into D^(t).
//
// Bound by latency: the rows and their copy are a few MB and mostly in L2.
// With one CTA per sequence, a warp taking its positions one after the other
// and one load at a time, a step of 16 sequences of 32 rows of 4096 spent
// 53 us here.
__global__ void __launch_bounds__(32 * kDriftRowsPerCta) drift_kernel(const DriftParams p) {
  grid_launch_dependents();  // every thread: the CTA counts once all of them have
  grid_dependency_wait();    // the previous step's drift kernel wrote prev
  const int row = blockIdx.x * kDriftRowsPerCta + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (row >= p.BP) return;
  const int nvec = p.H / 8;
  const uint4* cur = reinterpret_cast<const uint4*>(p.hidden + static_cast<size_t>(row) * p.H);
  uint4* prv = reinterpret_cast<uint4*>(p.prev + static_cast<size_t>(row) * p.H);
  float num = 0.0f, den = 0.0f;
  for (int v0 = lane; v0 < nvec; v0 += 32 * kDriftVecs) {
    uint4 x[kDriftVecs], y[kDriftVecs];
#pragma unroll
    for (int j = 0; j < kDriftVecs; ++j) {
      const int v = v0 + 32 * j;
      x[j] = v < nvec ? __ldg(cur + v) : make_uint4(0u, 0u, 0u, 0u);
      y[j] = v < nvec && p.t > 0 ? prv[v] : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int j = 0; j < kDriftVecs; ++j) {
      const __nv_bfloat16* xe = reinterpret_cast<const __nv_bfloat16*>(&x[j]);
      const __nv_bfloat16* ye = reinterpret_cast<const __nv_bfloat16*>(&y[j]);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float a = __bfloat162float(ye[i]);
        const float d = __bfloat162float(xe[i]) - a;
        num = fmaf(d, d, num);
        den = fmaf(a, a, den);
      }
      if (v0 + 32 * j < nvec) prv[v0 + 32 * j] = x[j];
    }
  }
  if (p.t == 0) return;
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    num += __shfl_xor_sync(0xffffffffu, num, off);
    den += __shfl_xor_sync(0xffffffffu, den, off);
  }
  const int b = row / p.P;
  unsigned done = 0;
  if (lane == 0) {
    p.ratio[row] = sqrtf(num) / sqrtf(den);
    __threadfence();
    done = atomicAdd(&p.count[b], 1u);
  }
  if (__shfl_sync(0xffffffffu, done, 0) != static_cast<unsigned>(p.P - 1)) return;
  __threadfence();
  float tot = 0.0f;
  for (int pp = lane; pp < p.P; pp += 32) tot += __ldcg(p.ratio + static_cast<size_t>(b) * p.P + pp);
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, off);
  if (lane == 0) {
    p.drift[(static_cast<size_t>(b) * p.n_blocks + p.blk) * p.T + p.t] = tot / static_cast<float>(p.P);
    p.count[b] = 0u;
  }
}

// ----------------------------------------------------------------- reset --

// The state of a new generation: byte-pattern fills of the context's arrays,
// each rounded up to 16 bytes (every buffer is padded to 256).  One launch
// instead of a memset per array, whose 19 launches of ~1.5 us each a toy-sized
// generation spent a tenth of its time on.
constexpr int kResetFills = 18;
constexpr int kResetThreads = 256;
struct ResetParams {
  uint4* ptr[kResetFills];
  unsigned long long vecs[kResetFills];  // 16-byte vectors
  uint32_t word[kResetFills];            // the pattern, 0 or ~0
};

__global__ void __launch_bounds__(kResetThreads) reset_state_kernel(const ResetParams p) {
  grid_launch_dependents();  // the first step's weight copies may start; it waits before the state
  for (int f = 0; f < kResetFills; ++f) {
    const uint32_t w = p.word[f];
    for (unsigned long long i = blockIdx.x * static_cast<unsigned long long>(kResetThreads) + threadIdx.x;
         i < p.vecs[f]; i += static_cast<unsigned long long>(gridDim.x) * kResetThreads)
      p.ptr[f][i] = make_uint4(w, w, w, w);
  }
}

// ------------------------------------------------- bounded-wait test hook --

// Waits, through the same bounded mbar_wait every step kernel uses, on a
// barrier nothing arrives at: after the wait limit it records `site` in the
// error word and returns (no trap, no fault; the context stays valid until
// the host reads the word).
__global__ void wait_timeout_probe_kernel(uint32_t* err, uint32_t site) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_wait(&bar, 0, &abort_flag, err, site);
}

// ------------------------------------------------------ list rebuild -----

struct ListParams {
  const int* tok;
  const int* exit_reason;
  int* list;
  int* row_of;
  int* d_M;
  int B, P, L, n_blocks, blk;
};

// Rebuild the masked-row list from the state (after a state upload).
__global__ void __launch_bounds__(kListThreads) rebuild_list_kernel(const ListParams p) {
  const int n = build_masked_list(p.tok, p.exit_reason, p.list, p.row_of, p.B, p.P, p.L,
                                  p.n_blocks, p.blk);
  if (threadIdx.x == 0) *p.d_M = n;
}

// ------------------------------------------ vocabulary-parallel head (shards) --

// A shard context holds the rows [v_off, v_off + V_shard) of W.  After its
// LM head, shard_rows_kernel reduces each masked row's partials into one
// triple (max * log2 e, sum of 2^(z log2 e - max), argmax as a global
// vocabulary index) in the exchange buffer; rows past M get the empty triple.
// Box 1's max, sum of exponentials and lowest-index argmax over the whole
// vocabulary are exact merges of these triples over the shards, which
// shard_merge_kernel does for every row before the commit.
constexpr int kShardThreads = 256;

struct ShardRowsParams {
  const float4* part;    // [rows, per_row] pair partials of this step (local indices)
  const float4* rowres;  // [rows] merged triple when the step wrote per-tile partials
  const int* d_M;
  float4* out;           // [rows_cap] exchange buffer
  int rows_cap;
  int n_pairs;           // the pair kernel's pairs
  int swap_max_n;        // its orientation rule
  int v_off;             // first vocabulary row of this shard
};

__global__ void __launch_bounds__(kShardThreads) shard_rows_kernel(const ShardRowsParams p) {
  grid_launch_dependents();  // every thread: the CTA counts once all of them have
  grid_dependency_wait();    // the pair kernel's partials (and the row merge's)
  const int M = *p.d_M;
  const int per_row = M > 0 ? pair_partials_per_row(M, p.n_pairs, pair_swapped(M, p.swap_max_n)) : 0;
  const int lane = threadIdx.x & 31;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < p.rows_cap; row += nw) {
    float m = kNegBig, s = 0.0f;
    int ix = INT_MAX;
    if (row < M) {  // the same in the whole warp
      const int n = per_row > 0 ? per_row : 1;
      const float4* pr = per_row > 0 ? p.part + static_cast<size_t>(row) * per_row : p.rowres + row;
      float4 q[kPartPerLane];  // every load in flight before the merge
#pragma unroll
      for (int u = 0; u < kPartPerLane; ++u)
        q[u] = lane + 32 * u < n ? __ldcg(pr + lane + 32 * u)
                                 : make_float4(kNegBig, 0.0f, __int_as_float(INT_MAX), 0.0f);
      for (int k = lane + 32 * kPartPerLane; k < n; k += 32) {
        const float4 a = __ldcg(pr + k);
        int i0 = __float_as_int(q[0].z);
        merge_tri(q[0].x, q[0].y, i0, a.x, a.y, __float_as_int(a.z));
        q[0].z = __int_as_float(i0);
      }
      __syncwarp();
      warp_merge(q, m, s, ix);
    }
    if (lane == 0)
      p.out[row] = make_float4(m, s, __int_as_float(ix == INT_MAX ? INT_MAX : ix + p.v_off), 0.0f);
  }
}

struct ShardMergeParams {
  const float4* gathered;  // [n_shards, rows_cap] every shard's exchange buffer, any order
  float4* rowres;          // [rows_cap] merged triple per row, read by the commit
  const int* d_M;
  int rows_cap, n_shards;
};

// One warp per masked row: the merge of the row's triples from every shard.
__global__ void __launch_bounds__(kShardThreads) shard_merge_kernel(const ShardMergeParams p) {
  grid_launch_dependents();  // every thread: the CTA counts once all of them have
  grid_dependency_wait();    // the previous commit's M and rowres readers
  const int M = *p.d_M;
  const int lane = threadIdx.x & 31;
  const int nw = (gridDim.x * blockDim.x) >> 5;
  for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < M; row += nw) {
    float m = kNegBig, s = 0.0f;
    int ix = INT_MAX;
    for (int k = lane; k < p.n_shards; k += 32) {
      const float4 a = __ldcg(p.gathered + static_cast<size_t>(k) * p.rows_cap + row);
      merge_tri(m, s, ix, a.x, a.y, __float_as_int(a.z));
    }
    __syncwarp();
    const float4 q[1] = {make_float4(m, s, __int_as_float(ix), 0.0f)};
    warp_merge(q, m, s, ix);
    if (lane == 0) p.rowres[row] = make_float4(m, s, __int_as_float(ix), 0.0f);
  }
}

// ------------------------------------------------------ merge + commit (K3) --

// One CTA per sequence: merge and commit of sequence blockIdx.x, then the
// last CTA to finish (atomic ticket; none needed for a single CTA) builds the
// next step's list and publishes the step.
__global__ void __launch_bounds__(kCommitThreads) merge_commit_kernel(const CommitParams p) {
  __shared__ int s_last;
  __shared__ CommitSmem cs;
  grid_launch_dependents();  // every thread: the CTA counts once all of them have
  // This step's M (d_M is rewritten only by the last CTA, after every CTA's
  // merge; at a block's first step every row is decoded) tells which LM-head
  // kernel decoded it: the pair kernel's tile partials were already merged
  // into one triple per row.  With prefetch_state, the kernel before this one
  // started only after the previous step had finished, so M and the
  // sequence's state are read before waiting for this step's partials.
  int M = 0;
  if (p.prefetch_state) {
    M = p.t == 0 ? p.B * p.P : __ldcg(p.d_M);
    commit_load(p, blockIdx.x, 1, cs);
  }
  // With prefetch_state the CTA starts when the first pair CTAs have left their
  // SMs (none fits beside one), while the last pairs end and the grid completes,
  // a few microseconds.  In them it makes a first pass over whatever the buffers
  // hold, writing nothing, so that the code (which the step's weight stream has
  // pushed out of the caches) is there when the second, real pass has to be
  // quick.  Blocks of eight steps without and with it: 66 rows, 4096 x 126464
  // 1269.5 -> 1265.2 us, 256 rows, 1024 x 22000 197.4 -> 192.6 us; within the
  // noise at 352 and 512 rows.
#pragma unroll 1
  for (int pass = p.prefetch_state ? 0 : 1; pass < 2; ++pass) {
    const bool real = pass == 1;
    if (real) grid_dependency_wait();  // partials of this step (and state of the previous one)
    if (!p.prefetch_state) {
      M = *p.d_M;
      commit_load(p, blockIdx.x, 1, cs);
    }
    const float4* part = p.part;
    int n_part = p.n_part;
    if (M >= p.pair_min_M) {
      n_part = pair_partials_per_row(M, p.pair_pairs, pair_swapped(M, p.pair_swap_max_n));
      if (n_part == 0) {
        part = p.rowres;
        n_part = 1;
      }
    }
    __syncthreads();  // cs
    merge_rows<kCommitPPW, false>(p, blockIdx.x, 1, cs, part, n_part, real);
    finish_sequences(p, blockIdx.x, 1, cs, real);
    if (gridDim.x > 1 && real) {
      if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicInc(p.ticket, gridDim.x - 1) == gridDim.x - 1;
      }
      __syncthreads();
      if (!s_last) return;
      __threadfence();
    }
    finish_step(p, -1, real);
  }
}

}  // namespace cai
