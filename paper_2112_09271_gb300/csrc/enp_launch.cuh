// What every launch site shares: the shared-memory limit of a kernel, and the status of
// launches.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>
#include <mutex>

namespace enp {

// The dynamic shared-memory limit of a kernel is a per-device attribute: each
// launch site keeps, per device, whether it has raised the limit (thread-safe).
struct SmemAttr {
  std::mutex mu;
  bool done[64] = {};
};
template <class K>
static cudaError_t raise_smem_limit(SmemAttr& st, K kern, size_t bytes) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64)
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  std::lock_guard<std::mutex> g(st.mu);
  if (st.done[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  // shared memory, not L1, bounds the resident blocks of these kernels
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess) st.done[dev] = true;
  return e;
}

// The status of a cudaLaunchKernelEx, and of the launches before it that were not
// asked for theirs. A failed launch also stays the thread's last error, and the next
// call to read that would report it as its own: it is taken here.
static inline cudaError_t launch_status(cudaError_t e) {
  const cudaError_t last = cudaGetLastError();
  return e != cudaSuccess ? e : last;
}

}  // namespace enp
