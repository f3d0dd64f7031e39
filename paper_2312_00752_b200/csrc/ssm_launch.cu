// What a launch needs to know about its kernel on the current device, asked once: the attribute and occupancy queries of
// one launch (two kernels weighed against each other, their shared-memory limits raised) took 10 us of host time a call.
#include <unordered_map>

#include "ssm_common.cuh"

namespace ssm {

namespace {
struct Key {
  const void* kernel;
  size_t smem;
  int device;
  bool operator==(const Key& o) const { return kernel == o.kernel && smem == o.smem && device == o.device; }
};
struct KeyHash {
  size_t operator()(const Key& k) const {
    return (reinterpret_cast<size_t>(k.kernel) >> 4) * 31 + k.smem * 17 + (size_t)k.device;
  }
};
}  // namespace

cudaError_t kernel_limits(const void* kernel, int threads, size_t smem, KernelLimits* out) {
  // one table per thread: no lock, and at most one entry per kernel, shared-memory size and device
  thread_local std::unordered_map<Key, KernelLimits, KeyHash> known;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const Key key{kernel, smem, dev};
  const auto it = known.find(key);
  if (it != known.end()) {
    *out = it->second;
    return cudaSuccess;
  }
  KernelLimits k{};
  if ((e = cudaDeviceGetAttribute(&k.sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if (smem > 0 && (e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k.per_sm, kernel, threads, smem)) != cudaSuccess) return e;
  if (k.per_sm < 1) return cudaErrorLaunchOutOfResources;
  known[key] = k;
  *out = k;
  return cudaSuccess;
}

}  // namespace ssm
