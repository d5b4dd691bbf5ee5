// Dynamic shared-memory limits of the kernels.
#pragma once

#include <cuda_runtime_api.h>

#include <cstddef>
#include <mutex>

namespace chdns {

// A kernel's dynamic shared-memory limit (and the non-portable cluster-size
// opt-in) as configured so far, on each device: the attribute belongs to the
// kernel in one device's context.  raise_smem_limit only ever raises it, under
// one lock for every kernel, so handles of different sizes driven from several
// host threads never leave a kernel below a size another one needs.
constexpr int kMaxDevices = 64;
struct SmemLimit {
  size_t bytes[kMaxDevices] = {};
  bool nonportable[kMaxDevices] = {};
};
inline std::mutex& kernel_attr_mutex() {
  static std::mutex m;
  return m;
}
template <typename K>
inline cudaError_t raise_smem_limit(K kernel, SmemLimit* lim, size_t smem, bool nonportable_cluster = false) {
  const void* f = reinterpret_cast<const void*>(kernel);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(kernel_attr_mutex());
  if (smem > lim->bytes[dev]) {
    e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    lim->bytes[dev] = smem;
  }
  if (nonportable_cluster && !lim->nonportable[dev]) {
    e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    lim->nonportable[dev] = true;
  }
  return cudaSuccess;
}

}  // namespace chdns
