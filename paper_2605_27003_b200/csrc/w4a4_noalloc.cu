// w4a4_quantize_noalloc: the activation-quantization step for callers that must not allocate.
//
// Some users of this library run where device allocation is off the table: inside a host callback, on
// a latency-critical path where a hidden cudaMalloc (which synchronises the device) is unacceptable, or
// inside a runtime that owns every byte of device memory through its own pool.  For them this one
// entry point runs the activation kernel without a context or a handle: its scratch (the reciprocal smoothing vector)
// lives in a fixed array that is part of the library image, and the caller supplies every input and output buffer.
#include "../../include/w4a4.h"

#include <cuda_runtime.h>

#include <mutex>

#include "quantize_kernel.cuh"

namespace {

constexpr int kNoAllocMaxK = 16384;                        // input channels
constexpr long long kNoAllocMaxElems = 4ll * 1024 * 1024;  // M * K
// The scratch itself: 64 KiB of device memory on every GPU that loads the library, held until
// the process exits.  In host code this name is only a stand-in; the device address is obtained once
// per device with cudaGetSymbolAddress below.
static __device__ __align__(256) float g_noalloc_rlam[kNoAllocMaxK];

constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
float* g_scratch_ptr[kMaxDevices] = {nullptr};

// Returns the device address of the scratch array on the current device (looked up once per device).
w4a4_status_t scratch_for_current_device(float** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return W4A4_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (g_scratch_ptr[dev] == nullptr) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_rlam) != cudaSuccess || p == nullptr) {
      cudaGetLastError();
      return W4A4_ERR_CUDA;
    }
    g_scratch_ptr[dev] = static_cast<float*>(p);
  }
  *out = g_scratch_ptr[dev];
  return W4A4_OK;
}

__global__ void noalloc_reciprocal_kernel(const float* __restrict__ lam, float* __restrict__ out, int K) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < K) out[k] = __fdiv_rn(1.0f, lam[k]);
}

}  // namespace

extern "C" w4a4_status_t w4a4_quantize_noalloc(const void* X, int M, int K, const float* lambda,
                                               const float* clip_table, int clip_index, int8_t* codes,
                                               float* scales, void* stream) {
  if (M < 0 || clip_index < 0) return W4A4_ERR_INVALID_ARG;
  if (K <= 0 || K % 64 != 0 || K > kNoAllocMaxK) return W4A4_ERR_SHAPE;
  if (static_cast<long long>(M) * K > kNoAllocMaxElems) return W4A4_ERR_SHAPE;  // beyond the built-in scratch
  if (M == 0) return W4A4_OK;
  if (!X || !lambda || !clip_table || !codes || !scales) return W4A4_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(X) & 15u) != 0) return W4A4_ERR_INVALID_ARG;

  float* rlam = nullptr;
  const w4a4_status_t st = scratch_for_current_device(&rlam);
  if (st != W4A4_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);

  // Every scratch byte that is read below is written first by this same call: nothing has to start at zero.
  noalloc_reciprocal_kernel<<<(K + 255) / 256, 256, 0, s>>>(lambda, rlam, K);
  w4a4::QuantizeParams p = {};
  p.X = static_cast<const uint16_t*>(X);
  p.M = M;
  p.K = K;
  p.rlam = rlam;
  p.clip_table = clip_table;
  p.clip_index = clip_index;
  p.codes = reinterpret_cast<uint8_t*>(codes);
  p.scales = scales;
  w4a4::QuantizePlan plan = w4a4::quantize_plan(M, K / 64, 0, 148, nullptr, 0, 0);
  constexpr int kSteps = 2;
  if (plan.steps != kSteps) plan.splits = (plan.splits + 1) / 2;
  const int cta_rows = w4a4::quantize_rows(kSteps, plan.warps), row_ctas = (M + cta_rows - 1) / cta_rows;
  p.row_warps = plan.warps;
  p.expand.first_cta = row_ctas;
  const CUtensorMap no_map = {};   // no low-rank branch
  w4a4::quantize_kernel<0, w4a4::kCodesInt8, kSteps>
      <<<dim3(row_ctas, plan.splits), w4a4::quantize_threads(0, plan.warps), w4a4::quantize_smem_bytes(0, kSteps, plan.warps, 1), s>>>(no_map, p);
  return cudaGetLastError() == cudaSuccess ? W4A4_OK : W4A4_ERR_CUDA;
}
