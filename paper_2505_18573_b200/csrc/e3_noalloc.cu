// e3_masked_mean_entropy_static: the masked mean entropy for callers that cannot hand over
// scratch memory.  The kernels of e3_masked_mean_entropy; the per-block partial sums live in an array that is part of the library image instead of a
// caller-provided workspace.  The paper has no counterpart for this entry point.
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "e3.h"
#include "e3_small.cuh"

namespace {

constexpr int kMaxBlocks = e3::kMeanBlocksMost;  // 1024 partials x 16 bytes = 16 KiB held by every device that loads the library
constexpr int kMaxDevices = 64;

struct Partial {
  double sum;
  double cnt;
};

// The scratch itself.  In host code this name is only a handle for the runtime's symbol
// table, never a device address: the address the kernels get comes from cudaGetSymbolAddress.
static __device__ __align__(256) Partial g_static_partials[kMaxBlocks];

std::mutex g_setup_lock;
Partial *g_device_scratch[kMaxDevices] = {};

// Device address of the scratch on the current device, looked up once per device.
cudaError_t scratch_for_current_device(Partial **out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> hold(g_setup_lock);
  if (!g_device_scratch[dev]) {
    Partial *p = nullptr;
    e = cudaGetSymbolAddress(reinterpret_cast<void **>(&p), g_static_partials);
    if (e != cudaSuccess) return e;
    if (!p) return cudaErrorInvalidSymbol;
    g_device_scratch[dev] = p;
  }
  *out = g_device_scratch[dev];
  return cudaSuccess;
}

inline bool off_boundary(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) != 0; }

}  // namespace

extern "C" e3_status e3_masked_mean_entropy_static(const float *ent, const uint8_t *mask, int64_t n,
                                                   double *out_mean, double *out_count, void *stream) {
  if (n < 0 || !out_mean || !out_count || (n > 0 && !ent)) return E3_ERR_INVALID_ARG;
  if (n > E3_STATIC_MEAN_MAX_TOKENS) return E3_ERR_WORKSPACE;  // beyond what the built-in scratch is sized for
  if (off_boundary(ent, 4) || off_boundary(out_mean, 8) || off_boundary(out_count, 8)) return E3_ERR_ALIGNMENT;
  Partial *scratch = nullptr;
  if (scratch_for_current_device(&scratch) != cudaSuccess) {
    (void)cudaGetLastError();
    return E3_ERR_CUDA;
  }
  // Every partial that is read has been written by the same call: nothing left behind by an earlier one can leak into it.
  return e3::launch_masked_mean(ent, mask, n, out_mean, out_count, scratch, false, static_cast<cudaStream_t>(stream)) == cudaSuccess
             ? E3_OK : E3_ERR_CUDA;
}
