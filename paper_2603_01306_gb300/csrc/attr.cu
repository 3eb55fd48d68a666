// A kernel's limit of dynamic shared memory belongs to the kernel and the
// device, not to the plan that asks for it: several host threads with plans of
// different sizes raise the same one.
#include <mutex>

#include "common.cuh"

namespace relax {

// Read and raise under one lock: two threads that both read the old limit could
// otherwise leave the smaller of their sizes, and the larger launch would be
// refused.
cudaError_t raise_smem(const void* kernel, size_t bytes) {
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  cudaFuncAttributes fa{};
  const cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e != cudaSuccess || fa.maxDynamicSharedSizeBytes >= (int)bytes) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace relax
