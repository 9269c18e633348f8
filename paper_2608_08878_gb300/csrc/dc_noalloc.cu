// dc_noalloc.cu -- full-cache decode attention for callers that cannot
// allocate device memory: the splits of a row merge through distributed shared
// memory (dc_full.cu), so that the call needs no device memory of its own.
//
// Which callers cannot allocate: runtimes that reserve all device memory up
// front and forbid further allocation (fixed-footprint serving processes),
// and latency-critical paths where an implicit device synchronisation from
// cudaMalloc/cudaFree is not acceptable. None of the handle-based calls fit
// them, because dc_cache_create allocates.
//
// The library's device code is loaded on a device at the first call there (lazy
// module loading): a caller that reserves the rest of device memory must make
// its first call before doing so.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <mutex>
#include <string>

#include "../../include/distillcache.h"
#include "dc_common.cuh"
#include "dc_kernels.h"

namespace {

// The limit on rows * group * (head_dim + 4) * 4 bytes (one split's partial
// results for every row), which once lived in an array of this size.
constexpr size_t kMaxPartialBytes = (size_t)16 << 20;  // 16 MiB

constexpr int kMaxDevices = 64;
std::mutex g_mu;
int g_num_sms[kMaxDevices] = {};

thread_local std::string g_noalloc_error;

dc_status noalloc_fail(dc_status s, const std::string& msg) {
  g_noalloc_error = msg;
  return s;
}

}  // namespace

extern "C" const char* dc_noalloc_last_error(void) { return g_noalloc_error.c_str(); }

extern "C" dc_status dc_attend_noalloc(const void* q, const void* k, const void* v, int rows, int n,
                                       int head_dim, int group, float* out, void* stream) {
  if (!q || !k || !v || !out) return noalloc_fail(DC_ERR_INVALID_ARG, "NULL pointer");
  if (head_dim != 64 && head_dim != 128) return noalloc_fail(DC_ERR_INVALID_ARG, "head_dim must be 64 or 128");
  if (group != 1 && group != 2 && group != 4 && group != 8)
    return noalloc_fail(DC_ERR_INVALID_ARG, "group must be 1, 2, 4 or 8");
  if (rows < 1 || rows > 65535 || n < 1) return noalloc_fail(DC_ERR_INVALID_ARG, "need 1 <= rows <= 65535 and n >= 1");
  if (((uintptr_t)k | (uintptr_t)v) & 15) return noalloc_fail(DC_ERR_INVALID_ARG, "k and v must be 16-byte aligned");
  const size_t per_split = (size_t)rows * group * (head_dim + 4) * sizeof(float);
  if (per_split > kMaxPartialBytes) {
    char buf[192];
    std::snprintf(buf, sizeof buf,
                  "rows * group * (head_dim + 4) * 4 = %zu bytes exceeds the %zu-byte scratch of the no-allocation path",
                  per_split, kMaxPartialBytes);
    return noalloc_fail(DC_ERR_CAPACITY, buf);
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return noalloc_fail(DC_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return noalloc_fail(DC_ERR_INVALID_ARG, "device ordinal out of range");
  int num_sms = 0;
  {
    // set-up, once per device, with that device current
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_num_sms[dev]) {
      int sms = 0;
      e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess)
        return noalloc_fail(DC_ERR_CUDA, std::string("cudaDeviceGetAttribute: ") + cudaGetErrorString(e));
      g_num_sms[dev] = sms;
    }
    num_sms = g_num_sms[dev];
  }

  dc::Dev p{};
  p.R = rows;
  p.cap = n;
  p.stride = n;
  p.d = head_dim;
  p.G = group;
  p.qh = group;  // q and out are [rows][group][head_dim]
  p.kvh = 1;
  p.K = const_cast<__nv_bfloat16*>(static_cast<const __nv_bfloat16*>(k));
  p.V = const_cast<__nv_bfloat16*>(static_cast<const __nv_bfloat16*>(v));
  p.c = (float)(1.4426950408889634 / std::sqrt((double)head_dim));
  if (!dc::launch_full_decode(p, n, num_sms, q, out, static_cast<cudaStream_t>(stream)))
    return noalloc_fail(DC_ERR_INVALID_ARG, "unsupported head_dim / group");
  e = cudaGetLastError();
  if (e != cudaSuccess) return noalloc_fail(DC_ERR_CUDA, std::string("launch: ") + cudaGetErrorString(e));
  return DC_OK;
}
