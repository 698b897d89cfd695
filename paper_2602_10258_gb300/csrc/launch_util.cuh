// Occupancy and device helpers shared by the launch code of several files.
#pragma once

#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <tuple>

#include "search_core.cuh"

namespace jag {

constexpr int kMaxCachedDevices = 64;

// SMs of the current device (read once per device).
inline int num_sms() {
  static std::mutex mu;
  static int sms[kMaxCachedDevices] = {};
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> g(mu);
  if (dev >= 0 && dev < kMaxCachedDevices && sms[dev] > 0) return sms[dev];
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  n = n > 0 ? n : 1;
  if (dev >= 0 && dev < kMaxCachedDevices) sms[dev] = n;
  return n;
}

// Blocks of `warps` warps of a kernel that fit on one SM of the current device
// with smem bytes of dynamic shared memory (0 if none).  The kernel's
// shared-memory limit is raised to the most the device gives it, so that
// launches of other sizes by other threads stay valid (again on each call for
// sizes that need it: a device reset forgets it); the answer is kept per
// (kernel, device, size): asking the runtime each time cost a small call up to
// 15 us on the host.
inline int blocks_per_sm_of(const void *kern, size_t smem, int warps) {
  static std::mutex mu;
  static std::map<std::tuple<const void *, int, size_t, int>, int> known;
  static std::map<std::pair<const void *, int>, int> limit;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> g(mu);
  const auto key = std::make_tuple(kern, dev, smem, warps);
  int &most = limit[std::make_pair(kern, dev)];
  const bool first = most == 0;
  if (first) {
    int optin = 0;
    cudaFuncAttributes fa{};
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaFuncGetAttributes(&fa, kern) != cudaSuccess)
      return 0;
    most = optin - (int)fa.sharedSizeBytes;
  }
  if (first || smem > 48 * 1024) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most) != cudaSuccess) return 0;
    // all of the unified L1 / shared storage may go to shared memory: the
    // occupancy query (and the launch) then count with the largest carve-out
    cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  }
  const auto it = known.find(key);
  if (it != known.end()) return it->second;
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, warps * 32, smem) != cudaSuccess) {
    cudaGetLastError();   // a size past the limit: no block fits
    b = 0;
  }
  if (known.size() >= 4096) known.clear();
  known[key] = b > 0 ? b : 0;
  return b > 0 ? b : 0;
}

template <class Kern>
inline int blocks_per_sm(Kern kern, size_t smem, int warps = kSearchWarps) {
  return blocks_per_sm_of(reinterpret_cast<const void *>(kern), smem, warps);
}

}  // namespace jag
