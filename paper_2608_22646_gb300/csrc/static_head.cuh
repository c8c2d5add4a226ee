// cai_head_rows_static: the decoding head (confidence and argmax of every
// row) for callers that cannot allocate device memory.
//
// Some callers cannot call cudaMalloc at the point where they need the head:
// code running while a memory pool owns the whole device, allocator-free
// inference runtimes that reserve all memory up front, or a caller inside a
// region where a new allocation would synchronise the device.  This entry point
// allocates nothing.  The caller passes its own weight, rows and outputs; the
// only scratch (the per-CTA softmax partials) is a fixed, file-scope device
// array that every GPU loading this library holds until the process exits.
//
// Kernels: the CTA-pair LM head (lm_head_pair_kernel, kStatic) reading the
// caller's row-major W in place, V cut evenly over the pairs, its partials in
// the static scratch; then one warp per row merges them.  Before, a single-CTA
// kernel of its own took 128-row tiles dealt out unevenly and loaded the rows
// as boxes of 16.
//
// Included once, at the end of cai.cu (it uses the device helpers of
// head_kernel.cuh, whose kernels must be defined in a single unit).
#pragma once

#include <atomic>
#include <mutex>

namespace cai {
namespace {

constexpr int kStaticMaxRows = 256;   // rows per call (one row tile)
constexpr int kStaticMaxParts = 160;  // partials per row: one per CTA
constexpr int kStaticStages = 6;      // ring slots of kPairStageBytes
constexpr int kStaticMaxDevices = 64;

// The whole scratch of the entry point: partial triples [row][CTA], plus one
// error word and the merge's ticket.  640 KiB + 256 bytes on every device that loads the library.
static __device__ __align__(256) float4 g_static_part[kStaticMaxRows * kStaticMaxParts];
static __device__ __align__(256) uint32_t g_static_err[64];

// One warp per row: merge the row's G partials, write c = 1 / S and the
// argmax.  If a bounded wait of the LM-head kernel gave up, every output is
// NaN / -1; the last CTA (err[1] is its ticket) then clears the error word for
// the next call.
__global__ void merge_rows_static_kernel(const float4* part, uint32_t* err, int M, int G,
                                         float* conf, int32_t* argmax) {
  grid_launch_dependents();  // the next call's set-up may overlap; it waits before it writes
  grid_dependency_wait();    // the LM head's partials
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const bool bad = __ldcg(err) != 0u;
  float m = kNegBig, s = 0.0f;
  int ix = INT_MAX;
  if (row < M) {  // the same in the whole warp
    float4 q[kStaticMaxParts / 32];  // every load in flight before the merge
#pragma unroll
    for (int u = 0; u < kStaticMaxParts / 32; ++u)
      q[u] = lane + 32 * u < G ? __ldcg(part + static_cast<size_t>(row) * G + lane + 32 * u)
                               : make_float4(kNegBig, 0.0f, __int_as_float(INT_MAX), 0.0f);
    warp_merge(q, m, s, ix);
  }
  if (lane == 0 && row < M) {
    const float c = row_confidence(m, s, ix);
    conf[row] = bad ? __int_as_float(0x7fc00000) : c;
    argmax[row] = bad ? -1 : ix;
  }
  __syncthreads();  // every warp of this CTA has read the error word
  if (threadIdx.x == 0 && atomicAdd(err + 1, 1u) == gridDim.x - 1) {
    err[0] = 0u;
    err[1] = 0u;
  }
}

typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                             const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                             const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct DeviceSetup {
  bool ready = false;
  float4* part = nullptr;
  uint32_t* err = nullptr;
  int pairs = 0;  // CTA pairs resident at once
  int stages = 0;
  size_t smem = 0;
};
std::mutex g_setup_mutex;
DeviceSetup g_setup[kStaticMaxDevices];
EncodeFn g_encode = nullptr;

// [1]: W read evict-first (pair_w_first).
void (*const static_kernels[2])(CUtensorMap, CUtensorMap, CUtensorMap, PairRowMaps, PairParams) = {
    lm_head_pair_kernel<false, true, false>, lm_head_pair_kernel<false, true, true>};

// Once per device, with that device current: the device addresses of the
// static scratch (a host-side name of a __device__ array is not a device
// address), the LM head's ring depth, shared-memory opt-in and resident pairs.
int setup_device(int dev, DeviceSetup** out) {
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  DeviceSetup& d = g_setup[dev];
  if (!d.ready) {
    if (!g_encode) {
      void* fn = nullptr;
      cudaDriverEntryPointQueryResult q;
      if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                           cudaEnableDefault, &q) != cudaSuccess ||
          q != cudaDriverEntryPointSuccess)
        return CAI_ERR_CUDA;
      g_encode = reinterpret_cast<EncodeFn>(fn);
    }
    int smem_optin = 0, sms = 0;
    cudaFuncAttributes attr{};
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&d.part), g_static_part) != cudaSuccess ||
        cudaGetSymbolAddress(reinterpret_cast<void**>(&d.err), g_static_err) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
            cudaSuccess ||
        cudaFuncGetAttributes(&attr, static_kernels[0]) != cudaSuccess) {
      cudaGetLastError();
      return CAI_ERR_CUDA;
    }
    d.stages = kStaticStages;
    while (d.stages > 2 &&
           pair_smem_bytes(d.stages, true) > static_cast<size_t>(smem_optin) - attr.sharedSizeBytes)
      --d.stages;
    d.smem = pair_smem_bytes(d.stages, true);
    cudaLaunchConfig_t qc = {};
    qc.gridDim = dim3(static_cast<unsigned>(sms & ~1));
    qc.blockDim = dim3(kPairThreads);
    qc.dynamicSmemBytes = d.smem;
    if (cudaFuncSetAttribute(static_kernels[0], cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(d.smem)) != cudaSuccess ||
        cudaFuncSetAttribute(static_kernels[1], cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(d.smem)) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&d.pairs, static_kernels[0], &qc) != cudaSuccess ||
        d.pairs < 1) {
      cudaGetLastError();
      return CAI_ERR_CUDA;
    }
    if (d.pairs > kStaticMaxParts / 2) d.pairs = kStaticMaxParts / 2;
    d.ready = true;
  }
  *out = &d;
  return CAI_OK;
}

bool encode(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(kBlockK), box_rows};
  cuuint32_t estr[2] = {1, 1};
  return g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Whether p is device (or managed) memory of device dev: the TMA maps and the
// kernels' stores must never be pointed at host memory.
bool on_device(const void* p, int dev) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged) && a.device == dev;
}

// Test hook: the next call makes its error word record a failed bounded wait
// before the merge (see cai_test_static_wait_timeout).
std::atomic<int> g_static_fail_next{0};

}  // namespace
}  // namespace cai

extern "C" int cai_head_rows_static(const void* W, int32_t V, int32_t H, const void* rows,
                                    int32_t M, float* conf, int32_t* argmax, void* stream) {
  using namespace cai;
  if (!W || !rows || !conf || !argmax) return CAI_ERR_ARG;
  if (M < 1 || M > kStaticMaxRows || V < 128 || H < 64 || H > 16384 || (H % 64) != 0)
    return CAI_ERR_SHAPE;
  if (reinterpret_cast<uintptr_t>(W) % 16 != 0 || reinterpret_cast<uintptr_t>(rows) % 16 != 0)
    return CAI_ERR_ARG;
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kStaticMaxDevices ||
      cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess) {
    cudaGetLastError();
    return CAI_ERR_CUDA;
  }
  if (major != 10 || minor != 3) return CAI_ERR_UNSUPPORTED;
  if (!on_device(W, dev) || !on_device(rows, dev) || !on_device(conf, dev) ||
      !on_device(argmax, dev))
    return CAI_ERR_ARG;
  DeviceSetup* d = nullptr;
  int r = setup_device(dev, &d);
  if (r != CAI_OK) return r;
  PairParams pp{};
  pp.th1 = pair_even_rows(V, d->pairs);
  pp.n_vt1 = (V + 2 * pp.th1 - 1) / (2 * pp.th1);
  const int pairs = pp.n_vt1 < d->pairs ? pp.n_vt1 : d->pairs;
  pp.part = d->part;
  pp.err = d->err;
  pp.V = V;
  pp.H = H;
  pp.n_vt = pp.n_vt1;
  pp.min_M = 1;
  pp.swap_max_n = pair_swap_width(H);
  pp.n_stages = d->stages;  // the ring of smem sized with the exchange buffer
  pp.ring_max = 8;
  pp.M_fixed = M;
  pp.w_dx = kPairBlockK;
  pp.w_ry = 1;
  const bool swap = pair_swapped(M, pp.swap_max_n);
  const int rows_box = swap ? swap_tile_cols(M, 1) / 2 : kPairHalf;
  CUtensorMap tm_w, tm_r;
  if (!encode(&tm_w, W, static_cast<uint64_t>(V), static_cast<uint64_t>(H), pp.th1) ||
      !encode(&tm_r, rows, static_cast<uint64_t>(M), static_cast<uint64_t>(H), rows_box))
    return CAI_ERR_ARG;
  PairRowMaps maps;
  for (CUtensorMap& m : maps.box) m = tm_r;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // An error left pending by earlier, unrelated work is not this call's.
  cudaGetLastError();
  // If the LM head did not launch, the merge would read a previous call's partials.
  if (launch_pdl(true, static_kernels[pair_w_first(V, H, true) ? 1 : 0], 2 * pairs, kPairThreads,
                 d->smem, s, tm_r, tm_w, tm_w, maps, pp) != cudaSuccess) {
    cudaGetLastError();
    return CAI_ERR_CUDA;
  }
  if (g_static_fail_next.exchange(0) != 0)
    wait_timeout_probe_kernel<<<1, 32, 0, s>>>(d->err, kErrWaitFull);
  const cudaError_t e =
      launch_pdl(true, merge_rows_static_kernel, (M + 7) / 8, 256, 0, s,
                 static_cast<const float4*>(d->part), d->err, static_cast<int>(M),
                 pair_partials_per_row(M, pairs, swap), conf, argmax);
  if (e != cudaSuccess || cudaGetLastError() != cudaSuccess) {
    cudaGetLastError();
    return CAI_ERR_CUDA;
  }
  return CAI_OK;
}

extern "C" int cai_test_static_wait_timeout(void) {
  cai::g_static_fail_next.store(1);
  return CAI_OK;
}
