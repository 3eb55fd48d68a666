// The library's stream-ordered scratch: one memory pool per device that keeps
// up to kKeep bytes between calls.  The default pool gives its memory back to
// the driver at every synchronisation, so each later call paid for mapping it
// again (about 190 us for the network's gradient step, 100 us for the
// standalone regularizer calls, when the caller synchronises in between).
// Allocation and release are ordered on the caller's stream, so the pool
// serves several threads and streams; it holds at most kKeep bytes beyond what
// is in use and gives them back when a handle is closed.
//
// On a stream that is being captured the allocation becomes a node whose memory
// the graph owns, so it is left to the default pool (making a pool there would
// also invalidate the capture).
#include <mutex>

#include "common.cuh"

namespace relax {

namespace {
constexpr int kMaxDevices = 64;
constexpr unsigned long long kKeep = 32ull << 20;
cudaMemPool_t g_pool[kMaxDevices] = {};
std::mutex g_mu;
}  // namespace

cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t st) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &capturing) == cudaSuccess && capturing != cudaStreamCaptureStatusNone)
    return cudaMallocAsync(p, bytes, st);
  cudaMemPool_t pool = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_pool[dev]) {
      cudaMemPoolProps props = {};
      props.allocType = cudaMemAllocationTypePinned;
      props.handleTypes = cudaMemHandleTypeNone;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      cudaMemPool_t made = nullptr;
      if ((e = cudaMemPoolCreate(&made, &props)) != cudaSuccess) return e;
      unsigned long long keep = kKeep;
      if ((e = cudaMemPoolSetAttribute(made, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
        cudaMemPoolDestroy(made);
        return e;
      }
      g_pool[dev] = made;
    }
    pool = g_pool[dev];
  }
  return cudaMallocFromPoolAsync(p, bytes, pool, st);
}

void pool_trim() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return;
  std::lock_guard<std::mutex> lock(g_mu);
  if (g_pool[dev]) cudaMemPoolTrimTo(g_pool[dev], 0);
}

}  // namespace relax
