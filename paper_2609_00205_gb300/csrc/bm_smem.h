// Dynamic shared memory beyond 48 KB: the limit a kernel is allowed is an
// attribute per device, not of the process.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace bm {

// Allows a kernel `bytes` of dynamic shared memory, once per device (done: the
// kernel's own mask of devices).  The same bytes every time, so host threads
// that meet here cannot lower each other's limit.
template <class F>
cudaError_t set_smem_once(F* fn, int bytes, std::atomic<unsigned>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned bit = dev < 32 ? 1u << dev : 0u;  // a device without a bit is set at each call
  if (done.load() & bit) return cudaSuccess;
  e = cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) done.fetch_or(bit);
  return e;
}

}  // namespace bm
