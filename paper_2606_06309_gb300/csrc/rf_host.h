// rf_host.h -- host-side helpers shared by the C-ABI translation units.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "rf.h"

namespace rf {

struct DeviceInfo {
  int device = -1;
  int sm_count = 0;
  int cc_major = 0;
  int cc_minor = 0;
  int max_smem_optin = 0;
  int l2_bytes = 0;
};

// Properties of the current device, cached per device ordinal (thread-safe).
rf_status current_device_info(DeviceInfo* out);

// Record a failure detail for rf_last_error() and return `st`.
rf_status fail(rf_status st, const char* what, cudaError_t err = cudaSuccess);

inline rf_status launch_status(const char* what) {
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? RF_OK : fail(RF_ERR_CUDA, what, e);
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// The argument errors of rf_attn, with nothing enqueued.
rf_status attn_check(const void* d_O, const void* d_Q, const void* d_K, const void* d_V,
                     int64_t qkv_row_stride, int64_t o_row_stride, int F, int N, int H, int d,
                     const int32_t* d_active, const int32_t* d_counts, float softmax_scale,
                     const void* d_workspace, int64_t workspace_bytes);

// Work that goes in front of an attention on its stream.
struct Front {
  rf_status (*launch)(const void* arg, cudaStream_t stream);
  const void* arg;
};

// rf_attn behind `front`, which is launched once nothing is left that could be refused: arguments
// checked, tensor maps made, kernel attributes set.
rf_status attn_behind(const Front& front, void* d_O, float* d_lse, const void* d_Q,
                      const void* d_K, const void* d_V, int64_t qkv_row_stride,
                      int64_t o_row_stride, int F, int N, int H, int d, const int32_t* d_active,
                      const int32_t* d_counts, float softmax_scale, void* d_workspace,
                      int64_t workspace_bytes, int32_t* d_status, rf_stream_t stream);

}  // namespace rf
