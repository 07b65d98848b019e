// Internals shared by the translation units of the library (not part of the C-ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "../../include/sdq.h"

namespace sdq {

// Sticky device-side flag words (one small allocation-free __device__ array per loaded library).
enum { FLAG_TIMEOUT = 1, FLAG_COUNT = 4 };

// device address of the flag words of the current device (nullptr on failure)
uint32_t* device_flags();

// Host-side facts about one device, looked up by the CURRENT device of the calling thread: they differ between the
// GPUs of one process (SM count; function attributes are per context), so nothing of this kind is a process-wide static.
// Threads share the table: sm_count is filled in under a lock, and so are pair_clusters, before clusters_known says so.
struct DeviceInfo {
  int sm_count;            // 0 until queried
  std::atomic<uint32_t> linear_attr;    // 1: the single-CTA GEMM instantiations carry their shared-memory attribute
  std::atomic<uint32_t> pair_attr;      // bit per CTA-pair GEMM instantiation
  std::atomic<uint32_t> diag_attr;      // the copy-rate diagnostic
  std::atomic<uint32_t> group_attr;     // the grouped few-token GEMM
  std::atomic<uint32_t> clusters_known; // 1: pair_clusters is filled in
  int pair_clusters[5];    // CTA-pair GEMM: clusters of k pairs that run at once
};
constexpr int MAX_DEVICES = 64;
// entry of device `dev` (0 <= dev < MAX_DEVICES) in the table; nullptr outside that range
DeviceInfo* device_info_slot(int dev);
// entry of the current device with sm_count filled in (nullptr on failure).  First use per device takes a lock.
DeviceInfo* device_info();

// status of a launch that returned `e`; takes the thread's last error with it, or the next call would report it as its own
inline sdq_status_t launch_status(cudaError_t e) {
  const cudaError_t last = cudaGetLastError();
  return e == cudaSuccess && last == cudaSuccess ? SDQ_OK : SDQ_ERR_CUDA;
}

// sdq_quantize_act; early_next: the next launch of the stream, the caller's own, may begin and read packed weights before this
// one has waited for its predecessor
sdq_status_t quantize_act(const void* X, int64_t M, int64_t K, int64_t ldx, const sdq_config_t* cfg, void* xq_buf, size_t xq_bytes, sdq_act_t* out,
                          void* stream, bool early_next);

}  // namespace sdq
