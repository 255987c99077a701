// Launch sizes.  Host code only.
#pragma once

#include <cuda_runtime_api.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

// What a launcher needs to know about a kernel on the current device, looked up once per kernel and device: the
// opt-in to its dynamic shared memory, which is an attribute of the kernel on one device, and the CTAs resident at
// once.  (The runtime queries cost more than the launch of a small grid.)
struct FitResidency {
  int per_sm = 0;  // CTAs per SM (0: not even one fits)
  int nsm = 0;     // SMs of the device
  long long ctas() const { return (long long)per_sm * nsm; }
};

// One table for the library, under its lock: launches come from several host threads.
struct FitResidencyTable {
  std::mutex mu;
  std::map<std::pair<const void*, int>, FitResidency> known;
};
inline FitResidencyTable& fit_residency_table() {
  static FitResidencyTable t;
  return t;
}

// count(&per_sm) answers the CTAs per SM of the kernel on the current device; it runs after the opt-in.
template <typename Count>
cudaError_t fit_residency(const void* kern, int smem, Count count, FitResidency* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  FitResidencyTable& t = fit_residency_table();
  std::lock_guard<std::mutex> lock(t.mu);
  const std::pair<const void*, int> key(kern, dev);
  auto it = t.known.find(key);
  if (it == t.known.end()) {
    FitResidency r;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&r.nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = count(&r.per_sm);
    if (e != cudaSuccess) return e;
    it = t.known.emplace(key, r).first;
  }
  *out = it->second;
  return cudaSuccess;
}

// the same with the runtime's occupancy query
inline cudaError_t fit_residency(const void* kern, int threads, int smem, FitResidency* out) {
  return fit_residency(
      kern, smem,
      [&](int* per_sm) {
        return cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(per_sm, kern, threads, smem, cudaOccupancyDefault);
      },
      out);
}

// Blocks that each system of a batch gets in a pass over all of them: per_sm blocks per SM shared by the batch, but at
// least `least` for every system (those of systems that have finished leave at once, and must not be all that the
// last ones have), and at most `most` (what the elements fill, what the pass's buffers hold).
inline long long fit_blocks_per_system(int per_sm, int nsm, int batch, int least, long long most) {
  return std::max(1LL, std::min(std::max((long long)least, (long long)per_sm * nsm / batch), most));
}
