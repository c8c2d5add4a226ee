// Online-softmax triples: (m, S, idx) with m the running maximum in log2 units,
// S = sum of 2^(z - m) over the values seen, idx the lowest index reaching m.
// Merging two triples or folding in one value is exact up to fp32 rounding, so
// any split of the vocabulary reduces to max_v z, sum_v exp(z_v - max) and the
// argmax (Box 1 of arXiv 2608.22646: c = exp(max - LSE) = 1 / S).
#pragma once

#include <climits>
#include <cstdint>
#include <cuda_bf16.h>

namespace cai {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kNegBig = -3.0e38f;  // "no logit yet": exp2(x - m) underflows to 0

// Sum of squares of eight bf16 values, in fp32 (the final RMSNorm's row
// statistic).
__device__ __forceinline__ float sumsq8(uint4 x) {
  const __nv_bfloat16* e = reinterpret_cast<const __nv_bfloat16*>(&x);
  float s = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float f = __bfloat162float(e[i]);
    s = fmaf(f, f, s);
  }
  return s;
}

// Final RMSNorm row scales 1 / sqrt(mean h^2 + eps) of rows [0, M) of the
// [M, H] bf16 rows `hid` into s_scale (shared memory), by the kWarps epilogue
// warps of an LM-head kernel (ew = 0.., each a whole warp; every one must
// call it), which then meet at named barrier 1: a row at a time per warp, 32
// lanes with eight 16-byte loads each in flight.
template <int kWarps>
__device__ __forceinline__ void epilogue_row_scales(const __nv_bfloat16* hid, int M, int H,
                                                    float eps, float* s_scale, int ew,
                                                    int lane) {
  const int nvec = H / 8;
  for (int r = ew; r < M; r += kWarps) {
    const uint4* src = reinterpret_cast<const uint4*>(hid + static_cast<size_t>(r) * H);
    float ss = 0.0f;
    for (int v0 = lane; v0 < nvec; v0 += 32 * 8) {
      uint4 x[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int v = v0 + 32 * j;
        x[j] = v < nvec ? __ldg(src + v) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) ss += sumsq8(x[j]);
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, off);
    if (lane == 0) s_scale[r] = rsqrtf(ss / static_cast<float>(H) + eps);
  }
  asm volatile("bar.sync 1, %0;" ::"n"(32 * kWarps) : "memory");  // the epilogue warps
}

__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Merge two online-softmax triples (m in log2 units, S = sum 2^(z - m), idx).
// The larger maximum keeps weight 1; ties keep the lower vocabulary index.
__device__ __forceinline__ void merge_tri(float& m, float& s, int& i, float mo, float so,
                                          int io) {
  const float e = fast_exp2(-fabsf(m - mo));
  const bool mine = m >= mo;
  const float sn = mine ? fmaf(so, e, s) : fmaf(s, e, so);
  const int in = (m > mo) ? i : ((mo > m) ? io : min(i, io));
  m = fmaxf(m, mo);
  s = sn;
  i = in;
}

__device__ __forceinline__ float warp_max(float x) {
  float y;
  asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(y) : "f"(x));
  return y;
}

// Merge kN triples of every lane over the whole warp (converged); every lane
// gets the result, as a sequence of merge_tri would give it up to fp32
// rounding.  The maximum comes first, in one warp reduction, so that no
// exponential waits for another: a tree of merge_tri is five of them one
// after the other.
template <int kN>
__device__ __forceinline__ void warp_merge(const float4 (&q)[kN], float& m, float& s, int& ix) {
  m = q[0].x;
#pragma unroll
  for (int u = 1; u < kN; ++u) m = fmaxf(m, q[u].x);
  m = warp_max(m);
  s = 0.0f;
  ix = INT_MAX;
#pragma unroll
  for (int u = 0; u < kN; ++u) {
    s = fmaf(q[u].y, fast_exp2(q[u].x - m), s);
    ix = q[u].x == m ? min(ix, __float_as_int(q[u].z)) : ix;
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  ix = __reduce_min_sync(0xffffffffu, ix);
}

// A row's confidence max_v p_v = exp(m - LSE) = 1 / S from its merged triple.  A
// row without a logit above the empty maximum (all NaN or -inf) has no softmax:
// its confidence is NaN, which passes no threshold, and its index 0, the lowest
// of the equal ones, so that what is stored as an argmax always is one.  (A +inf
// logit makes S, and so the confidence, NaN by itself: exp2(inf - inf).)
__device__ __forceinline__ float row_confidence(float m, float s, int& ix) {
  if (m > kNegBig) return 1.0f / s;
  ix = 0;
  return __int_as_float(0x7fc00000);
}

// 32 lanes x 32 columns of online-softmax triples -> lane l holds the merge of
// column l over the 32 lanes, in m[0], s[0], ix[0].  Five halving steps: at
// width w each lane keeps half of its live columns and receives the partner's
// copy of the same columns (31 merges per lane, one exponential each).
__device__ __forceinline__ void transpose_merge32(float (&m)[32], float (&s)[32], int (&ix)[32],
                                                  int lane) {
#pragma unroll
  for (int w = 16; w >= 1; w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int c = 0; c < w; ++c) {
      float km = up ? m[c + w] : m[c];
      float ks = up ? s[c + w] : s[c];
      int ki = up ? ix[c + w] : ix[c];
      const float sm = up ? m[c] : m[c + w];
      const float ss = up ? s[c] : s[c + w];
      const int si = up ? ix[c] : ix[c + w];
      const float rm = __shfl_xor_sync(0xffffffffu, sm, w);
      const float rs = __shfl_xor_sync(0xffffffffu, ss, w);
      const int ri = __shfl_xor_sync(0xffffffffu, si, w);
      merge_tri(km, ks, ki, rm, rs, ri);
      m[c] = km;
      s[c] = ks;
      ix[c] = ki;
    }
  }
}

// Fold the logits z (log2 units) of vocabulary rows vrow, vrow + 8, vrow + 16,
// vrow + 24 into a running triple.  Rows arrive in increasing order, so only a
// strictly larger value replaces the argmax.
__device__ __forceinline__ void fold4(float& m, float& s, int& ix, const float (&z)[4], int vrow) {
  const float mx = fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3]));
  const int k = z[0] == mx ? 0 : z[1] == mx ? 8 : z[2] == mx ? 16 : 24;
  const float mn = fmaxf(m, mx);
  const float add = (fast_exp2(z[0] - mn) + fast_exp2(z[1] - mn)) +
                    (fast_exp2(z[2] - mn) + fast_exp2(z[3] - mn));
  s = fmaf(s, fast_exp2(m - mn), add);
  ix = mx > m ? vrow + k : ix;
  m = mn;
}

// Four columns' triples of each thread (index 2 j + e), the same columns in
// the eight lanes that agree in bits 0 and 1: merge over those lanes; lane l
// is left with the column j = bit 4, e = bit 3 of l (both values of bit 2 hold
// it).
__device__ __forceinline__ void merge_frag8(const float* m, const float* s, const int* ix, int lane,
                                            float4& out) {
  const bool up16 = (lane & 16) != 0, up8 = (lane & 8) != 0;
  float am[2], as[2];
  int ai[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    am[e] = up16 ? m[2 + e] : m[e];
    as[e] = up16 ? s[2 + e] : s[e];
    ai[e] = up16 ? ix[2 + e] : ix[e];
    const float rm = __shfl_xor_sync(0xffffffffu, up16 ? m[e] : m[2 + e], 16);
    const float rs = __shfl_xor_sync(0xffffffffu, up16 ? s[e] : s[2 + e], 16);
    const int ri = __shfl_xor_sync(0xffffffffu, up16 ? ix[e] : ix[2 + e], 16);
    merge_tri(am[e], as[e], ai[e], rm, rs, ri);
  }
  float km = up8 ? am[1] : am[0], ks = up8 ? as[1] : as[0];
  int ki = up8 ? ai[1] : ai[0];
  {
    const float rm = __shfl_xor_sync(0xffffffffu, up8 ? am[0] : am[1], 8);
    const float rs = __shfl_xor_sync(0xffffffffu, up8 ? as[0] : as[1], 8);
    const int ri = __shfl_xor_sync(0xffffffffu, up8 ? ai[0] : ai[1], 8);
    merge_tri(km, ks, ki, rm, rs, ri);
  }
  const float rm = __shfl_xor_sync(0xffffffffu, km, 4);
  const float rs = __shfl_xor_sync(0xffffffffu, ks, 4);
  const int ri = __shfl_xor_sync(0xffffffffu, ki, 4);
  merge_tri(km, ks, ki, rm, rs, ri);
  out = make_float4(km, ks, __int_as_float(ki), 0.0f);
}

// Fold 32 logits x[k] of one row (times the scale rs, which includes log2 e),
// vocabulary rows v0 + k, of which the first nvalid exist (the same number in
// every thread of the warp), into a running triple.  The index is searched for
// only when the maximum moves, which after the first few chunks it rarely does.
__device__ __forceinline__ void fold_row32(float& m, float& s, int& ix, const uint32_t (&x)[32],
                                           float rs, int v0, int nvalid) {
  float z[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) z[k] = __fmul_rn(__uint_as_float(x[k]), rs);
  if (nvalid < 32) {
#pragma unroll
    for (int k = 0; k < 32; ++k) z[k] = k < nvalid ? z[k] : -INFINITY;
  }
  float t[4] = {z[0], z[1], z[2], z[3]};
#pragma unroll
  for (int k = 4; k < 32; ++k) t[k & 3] = fmaxf(t[k & 3], z[k]);
  const float cm = fmaxf(fmaxf(t[0], t[1]), fmaxf(t[2], t[3]));
  if (cm > m) {  // strictly: an equal maximum keeps the lower index
    s *= fast_exp2(m - cm);
    m = cm;
    int ci = 0;
#pragma unroll
    for (int k = 31; k >= 0; --k) ci = z[k] == cm ? k : ci;
    ix = v0 + ci;
  }
  float c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int k = 0; k < 32; ++k) c[k & 3] += fast_exp2(z[k] - m);
  s += (c[0] + c[1]) + (c[2] + c[3]);
}

// 32 rows (one per lane) x 32 columns of logits -> lane l holds the
// (max, sum, argmax) of column l over the 32 rows.  Column c's logits are
// scaled by log2 e, times col_scale[c] when given (a per-row normalisation
// of the decoded hidden states, see lm_head_softmax_kernel; global or shared
// memory).
__device__ __forceinline__ void transpose_reduce32(const uint32_t (&v)[32], bool valid, int vrow,
                                                   int lane, float& om, float& os, int& oi,
                                                   const float* col_scale = nullptr) {
  float m[32], s[32];
  int ix[32];
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    const float sc = col_scale ? kLog2e * col_scale[c] : kLog2e;
    m[c] = valid ? __uint_as_float(v[c]) * sc : kNegBig;
    s[c] = valid ? 1.0f : 0.0f;
    ix[c] = valid ? vrow : INT_MAX;
  }
  transpose_merge32(m, s, ix, lane);
  om = m[0];
  os = s[0];
  oi = ix[0];
}

// Fold one logit z (log2 units) of vocabulary row `row` into a running
// triple.  Rows arrive in increasing order, so only a strictly larger value
// replaces the argmax (ties keep the lower index).
__device__ __forceinline__ void online_update(float& m, float& s, int& i, float z, int row) {
  const float d = z - m;
  const float e = fast_exp2(-fabsf(d));
  const bool up = d > 0.0f;
  s = up ? fmaf(s, e, 1.0f) : s + e;
  m = up ? z : m;
  i = up ? row : i;
}

}  // namespace cai
