// The commit rule of CAI-dLLM (arXiv 2608.22646, Algorithm 1 with Boxes 2-7)
// for one sequence, run by one CTA, and the end-of-step bookkeeping (the next
// step's masked-row list and the host-visible record).  Shared by the merge
// kernel of the multi-kernel step and by the single-kernel step, whose last
// LM-head CTA runs it.
#pragma once

#include <cstdint>

#include "ptx.cuh"
#include "softmax.cuh"

namespace cai {

constexpr int kMask = -1;
enum : int { kRunning = 0, kExitDone = 1, kExitGrind = 2, kExitTmax = 3 };
enum : uint32_t {
  kFlagGating = 1u,
  kFlagPosFactor = 2u,
  kFlagFlush = 4u,
  kFlagQuarterPos = 8u,
  kFlagQuarterBlocks = 16u,
  kFlagDiag = 128u
};
constexpr int kMaxP = 256;
constexpr int kPosPerWarp = 6;   // positions whose partials a warp loads at once
constexpr int kPartPerLane = 5;  // partial slots a lane loads per position (G <= 160)

// Host-visible record of the last committed step, one 64-bit word in mapped
// pinned memory written by a single store (so the host never sees a torn
// record): bits 0-31 step id + 1, bit 32 every sequence has exited the block,
// bit 33 the device error word is non-zero, bits 34-48 the block index.
struct HostFlag {
  unsigned long long word;  // 0 = no step committed yet
  unsigned long long pad;
};
__host__ __device__ inline unsigned long long host_flag_word(int step_id, bool all_done, bool err,
                                                             int blk) {
  return static_cast<unsigned long long>(static_cast<uint32_t>(step_id) + 1u) |
         (static_cast<unsigned long long>(all_done ? 1u : 0u) << 32) |
         (static_cast<unsigned long long>(err ? 1u : 0u) << 33) |
         (static_cast<unsigned long long>(static_cast<uint32_t>(blk) & 0x7FFFu) << 34);
}

struct StateArrays {
  int* tok;
  float* conf;
  float* s0;
  uint8_t* budget;
  int16_t* cstep;
  int* cand;
  int* ell;
  int* eta;
  int* exit_reason;
  int* exit_step;
  int* unresolved;
  int* m_hist;
  uint8_t* run;     // diagnostics: consecutive decoded steps with the same argmax
  int16_t* stable;  // diagnostics: stability step t_i^*, -1
  float* drift;     // diagnostics: [B, n_blocks, T] relative drift D^(t)
};

struct CommitParams {
  const float4* part;     // [rows, n_part] softmax partials of this step
  int n_part;             // partial slots per row (one per LM-head CTA)
  const float4* rowres;   // [rows] merged triple per row when the pair kernel decoded the step
  int pair_min_M;         // steps with at least this many rows ran the pair kernel
  int pair_pairs;         // pairs of the pair kernel's grid
  int pair_swap_max_n;    // the pair kernel's orientation rule (pair_swapped)
  int identity_rows;      // 1: row of (b, p) is b P + p; 0: row_of[b P + p]
  int prefetch_state;     // merge kernel: read the sequence's state before waiting for the
                          // LM head (the kernel before it starts only after its own wait)
  StateArrays st;
  int* list;
  int* row_of;
  int* d_M;
  int* m_hist_slot;       // this step's M_t (written by the single-kernel step)
  unsigned* ticket;       // zero between steps that use it (atomicInc wraps it)
  unsigned long long* pub;  // (step id + 1) << 32 | masked rows left, written by finish_step
  HostFlag* hf;           // device alias of the mapped host record
  uint32_t* err;
  int B, P, L, n_blocks, T, blk, t, step_id;
  int K;
  int eta_mode;           // 0 count, 1 fraction of the generation length
  float eta_bar;
  float theta_fb;
  int budget_half;        // Box 5 "p < 32" tier boundary
  int budget_late;        // Box 5 "p >= 48" tier boundary
  uint32_t flags;
  float theta_tab[kMaxP]; // theta_i(t) per position (Box 6), from the host
};

__device__ __forceinline__ int budget_tier(float s, int p, int half, int late) {
  if (s > 0.50f && p < half) return 8;
  if (s < 0.25f || p >= late) return 64;
  return 32;
}

// Working set of one commit, in shared memory the caller provides (the LM-head
// kernel lends its drained W ring): the block's positions of one or several
// sequences, at most kMaxP of them, sequence by sequence.
struct CommitSmem {
  int tok[kMaxP];      // token after this step (kMask while masked)
  int cand[kMaxP];     // diagnostics: argmax of the previous decoded step
  float conf[kMaxP];   // confidence and argmax of this step (merge_rows)
  int idx[kMaxP];
  int row[kMaxP];      // partial row of the position in this step (masked positions)
  uint8_t bud[kMaxP];  // budget before this step
  uint8_t run[kMaxP];  // diagnostics: same-argmax run before this step
  int16_t stable[kMaxP];  // diagnostics: stability step before this step
  // per sequence
  int running[kMaxP];  // the sequence has not left the block
  int ell[kMaxP];      // low-yield counter before this step
  int eta[kMaxP], left[kMaxP], unres[kMaxP], reason[kMaxP];  // this step's counts and exit
  int decoded, remaining;  // over all sequences: rows decoded, rows still masked afterwards
};

// Reads what one step of Algorithm 1 needs of the state of sequences [b0, b0 +
// nb) into cs, in one round of loads by the whole calling CTA (visible to it
// after its next __syncthreads): the block's tokens and budgets, the exit
// state, ell, and the partial row of every position.  All of it was written by
// the previous step's commit (or by the reset) except, at a block's first step,
// the row list, which the gather then makes the identity; so a commit that
// follows an LM head which itself waited for the previous step may read it
// before waiting for the partials.
__device__ __forceinline__ void commit_load(const CommitParams& p, int b0, int nb, CommitSmem& cs) {
  const int tid = threadIdx.x;
  for (int q = tid; q < nb; q += blockDim.x) {
    cs.running[q] = __ldcg(&p.st.exit_reason[(b0 + q) * p.n_blocks + p.blk]) == kRunning;
    cs.ell[q] = __ldcg(&p.st.ell[b0 + q]);
    cs.eta[q] = cs.left[q] = cs.unres[q] = 0;
    cs.reason[q] = kRunning;
  }
  if (tid == 0) cs.decoded = cs.remaining = 0;
  const bool diag = (p.flags & kFlagDiag) != 0;
  const bool ident = p.identity_rows || p.t == 0;
  for (int i = tid; i < nb * p.P; i += blockDim.x) {
    const int q = i / p.P;
    const size_t g = static_cast<size_t>(b0 + q) * p.L + p.blk * p.P + (i - q * p.P);
    cs.tok[i] = __ldcg(&p.st.tok[g]);
    cs.bud[i] = __ldcg(&p.st.budget[g]);
    cs.row[i] = ident ? b0 * p.P + i : __ldcg(&p.row_of[b0 * p.P + i]);
    if (diag) {
      cs.cand[i] = __ldcg(&p.st.cand[g]);
      cs.run[i] = __ldcg(&p.st.run[g]);
      cs.stable[i] = __ldcg(&p.st.stable[g]);
    }
  }
}

// The commit rule (Box 6, Eq. position_commit, with the step-zero init of Boxes
// 2 and 5) for position i of cs with confidence c and argmax ix, by one thread.
__device__ __forceinline__ void commit_position(const CommitParams& p, int b0, CommitSmem& cs,
                                                int i, float c, int ix) {
  const int sq = i / p.P, pp = i - sq * p.P;
  const size_t g = static_cast<size_t>(b0 + sq) * p.L + p.blk * p.P + pp;
  int bud = cs.bud[i];
  if (p.t == 0) {
    bud = budget_tier(c, pp, p.budget_half, p.budget_late);
    p.st.s0[g] = c;
    p.st.budget[g] = static_cast<uint8_t>(bud);
  }
  if ((p.flags & kFlagDiag) != 0) {
    // Section 2.1: stable once the argmax has held for three decoded steps.
    const int run = (p.t > 0 && cs.cand[i] == ix) ? cs.run[i] + 1 : 1;
    p.st.run[g] = static_cast<uint8_t>(run < 255 ? run : 255);
    if (run >= 3 && cs.stable[i] < 0) p.st.stable[g] = static_cast<int16_t>(p.t);
  }
  p.st.conf[g] = c;
  p.st.cand[g] = ix;
  cs.conf[i] = c;
  cs.idx[i] = ix;
  const bool by_conf = c >= p.theta_tab[pp];
  const bool by_budget = (p.flags & kFlagGating) != 0 && p.t >= bud;
  if (by_conf || by_budget) {
    cs.tok[i] = ix;
    p.st.tok[g] = ix;
    p.st.cstep[g] = static_cast<int16_t>(p.t);
    atomicAdd(&cs.eta[sq], 1);
  } else {
    atomicAdd(&cs.left[sq], 1);
  }
}

// Merges the partials of the block's positions of sequences [b0, b0 + nb) (nb P
// <= kMaxP), by the whole calling CTA (blockDim.x a multiple of 32): a warp per
// position, kPPW at a time, all loads issued before any merge.  kAll: every
// position, in the order of the block (rows of a single-kernel step), into
// cs.conf and cs.idx, which needs no state.  Else the still-masked positions of
// running sequences, at the rows commit_load has read, each committed by its
// warp's first lane as soon as it is merged (a second pass with a thread per
// position cost 0.8 to 1.2 us a step).  With `real` false nothing outside the
// CTA is written and cs is left alone: a pass over stale partials that brings
// the code into the instruction caches.
template <int kPPW, bool kAll>
__device__ void merge_rows(const CommitParams& p, int b0, int nb, CommitSmem& cs,
                           const float4* part, int n_part, bool real = true) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nwarps = blockDim.x >> 5;
  const int n = nb * p.P;
  for (int base = warp; base < n; base += nwarps * kPPW) {
    int row[kPPW];
    float4 q[kPPW][kPartPerLane];
#pragma unroll
    for (int j = 0; j < kPPW; ++j) {
      const int i = base + j * nwarps;
      row[j] = -1;
      if (kAll) {
        if (i < n) row[j] = b0 * p.P + i;
      } else if (i < n && cs.tok[i] == kMask && cs.running[i / p.P]) {
        row[j] = cs.row[i];
        if (!CAI_IN_RANGE(row[j] < p.B * p.P, p.err)) row[j] = -2;
        if (row[j] < 0) {
          if (lane == 0 && real) atomicOr(p.err, kErrBadRow);
          row[j] = -2;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < kPPW; ++j) {
      const float4* pr = part + static_cast<size_t>(row[j] < 0 ? 0 : row[j]) * n_part;
#pragma unroll
      for (int u = 0; u < kPartPerLane; ++u) {
        const int k = lane + 32 * u;
        q[j][u] = (row[j] >= 0 && k < n_part)
                      ? __ldcg(pr + k)
                      : make_float4(kNegBig, 0.0f, __int_as_float(INT_MAX), 0.0f);
      }
    }
#pragma unroll
    for (int j = 0; j < kPPW; ++j) {
      if (row[j] < 0) continue;  // warp-uniform
      for (int k = lane + 32 * kPartPerLane; k < n_part; k += 32) {
        const float4 r = __ldcg(part + static_cast<size_t>(row[j]) * n_part + k);
        int i0 = __float_as_int(q[j][0].z);
        merge_tri(q[j][0].x, q[j][0].y, i0, r.x, r.y, __float_as_int(r.z));
        q[j][0].z = __int_as_float(i0);
      }
      __syncwarp();
      float m, s;
      int ix;
      warp_merge(q[j], m, s, ix);
      const int i = base + j * nwarps;
      const float c = row_confidence(m, s, ix);
      if (lane == 0) {
        if (kAll) {
          cs.conf[i] = c;
          cs.idx[i] = ix;
        } else if (real) {
          commit_position(p, b0, cs, i, c, ix);
        }
      }
    }
  }
}

// The end of a step of Algorithm 1 for the sequences [b0, b0 + nb) once their
// positions are committed (commit_position), by the whole calling CTA; every
// thread must call it.  One thread per sequence updates the low-yield counter
// and the exit state (Box 7, Algorithm 1).  Global state is only written, never
// re-read.  Leaves in cs, for every thread, the positions decoded and those
// still masked afterwards in running sequences.  `real` as in merge_rows.
__device__ void finish_sequences(const CommitParams& p, int b0, int nb, CommitSmem& cs,
                                 bool real = true) {
  const int tid = threadIdx.x;
  const int n = nb * p.P;
  const bool gating = (p.flags & kFlagGating) != 0;
  __syncthreads();
  if (!real) return;
  bool exits = false;
  for (int q = tid; q < nb; q += blockDim.x) {
    if (!cs.running[q]) continue;
    const int eta = cs.eta[q];
    p.st.eta[b0 + q] = eta;
    const bool low = p.eta_mode == 1
                         ? (static_cast<double>(eta) / (static_cast<double>(p.n_blocks) * p.P) <
                            static_cast<double>(p.eta_bar))
                         : (static_cast<float>(eta) < p.eta_bar);
    // Algorithm 1 sets ell <- 0 before the block's first step.
    const int ell = low ? (p.t == 0 ? 0 : cs.ell[q]) + 1 : 0;
    p.st.ell[b0 + q] = ell;
    int reason = kRunning;
    if (gating && ell >= p.K)
      reason = kExitGrind;
    else if (cs.left[q] == 0)
      reason = kExitDone;
    else if (p.t == p.T - 1)
      reason = kExitTmax;
    cs.reason[q] = reason;
    atomicAdd(&cs.decoded, eta + cs.left[q]);
    if (reason == kRunning)
      atomicAdd(&cs.remaining, cs.left[q]);
    else
      exits = true;
  }
  if (!__syncthreads_or(exits)) return;
  for (int i = tid; i < n; i += blockDim.x) {
    const int sq = i / p.P;
    const int reason = cs.reason[sq];
    if (reason == kRunning || cs.tok[i] != kMask) continue;
    const size_t g = static_cast<size_t>(b0 + sq) * p.L + p.blk * p.P + (i - sq * p.P);
    if ((reason == kExitGrind && cs.conf[i] > p.theta_fb) || (p.flags & kFlagFlush)) {
      p.st.tok[g] = cs.idx[i];
      p.st.cstep[g] = static_cast<int16_t>(p.t);
    } else {
      atomicAdd(&cs.unres[sq], 1);
    }
  }
  __syncthreads();
  for (int q = tid; q < nb; q += blockDim.x) {
    if (cs.reason[q] == kRunning) continue;
    const int eb = (b0 + q) * p.n_blocks + p.blk;
    p.st.exit_reason[eb] = cs.reason[q];
    p.st.exit_step[eb] = p.t;
    p.st.unresolved[eb] = cs.unres[q];
  }
  __syncthreads();
}

// Compact, in (b, p) order, the still-masked tokens of running sequences of
// block blk into list / row_of; returns the count.  One CTA (blockDim.x a
// multiple of 32, at most 1024).  Reads bypass L1: other CTAs wrote this state.
__device__ int build_masked_list(const int* tok, const int* exit_reason, int* list, int* row_of,
                                 int B, int P, int L, int n_blocks, int blk, bool real = true) {
  __shared__ int s_wsum[32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nwarps = blockDim.x >> 5;
  const int BP = B * P;
  int base = 0;
  for (int i0 = 0; i0 < BP; i0 += blockDim.x) {
    const int i = i0 + tid;
    bool mk = false;
    if (i < BP) {
      // Both loads issued before either is tested (one round trip, not two).
      const int b = i / P, pp = i - b * P;
      const int tk = __ldcg(&tok[static_cast<size_t>(b) * L + blk * P + pp]);
      const int ex = __ldcg(&exit_reason[b * n_blocks + blk]);
      mk = (tk == kMask) & (ex == kRunning);
    }
    const unsigned bal = __ballot_sync(0xffffffffu, mk);
    const int wpre = __popc(bal & ((1u << lane) - 1u));
    if (lane == 0) s_wsum[warp] = __popc(bal);
    __syncthreads();
    int woff = 0, tot = 0;
    for (int w = 0; w < nwarps; ++w) {
      const int c = s_wsum[w];
      woff += (w < warp) ? c : 0;
      tot += c;
    }
    if (i < BP && real) {
      if (mk) {
        list[base + woff + wpre] = i;
        row_of[i] = base + woff + wpre;
      } else {
        row_of[i] = -1;
      }
    }
    base += tot;
    __syncthreads();
    if (!real) break;
  }
  return base;
}

// End of a step, by the last CTA: the next step's list (multi-kernel step
// only; the single-kernel step decodes every row and needs none), M_{t+1},
// and the host-visible record.  `remaining` is the masked
// count of running sequences when the caller already knows it (-1: count).
// `real` as in merge_rows.
__device__ void finish_step(const CommitParams& p, int remaining = -1, bool real = true) {
  const int n = remaining >= 0 ? remaining
                               : build_masked_list(p.st.tok, p.st.exit_reason, p.list, p.row_of,
                                                   p.B, p.P, p.L, p.n_blocks, p.blk, real);
  if (threadIdx.x == 0 && real) {
    *p.d_M = n;
    const bool err = *reinterpret_cast<volatile uint32_t*>(p.err) != 0u;
    // The host uses this word only for control flow; it reads the state
    // itself through stream-ordered copies, so no system fence is needed.
    *reinterpret_cast<volatile unsigned long long*>(&p.hf->word) =
        host_flag_word(p.step_id, n == 0, err, p.blk);
    // Device copy for the next step, which may already be running (see the
    // LM-head kernel): it stops early when this step left nothing masked.
    *reinterpret_cast<volatile unsigned long long*>(p.pub) =
        (static_cast<unsigned long long>(static_cast<uint32_t>(p.step_id + 1)) << 32) |
        static_cast<uint32_t>(n);
  }
}

}  // namespace cai
