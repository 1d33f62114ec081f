// Device scratch of the kernel-level entry points (partial sums, digit planes,
// the eigensolver's work matrices), taken in stream order from a memory pool of
// this library, one per device.
//
// The device's default pool gives everything back at each synchronisation of a
// stream, so a caller that waits for its result pays for a fresh mapping on the
// next call (about 200 us at any size: 651 us alone against 431 us in a row for
// the residual of 262,144 x 71).  This pool keeps at most kKeep bytes a device;
// what lies above goes back at the next synchronisation, and lobpcg_destroy,
// lobpcg_chebyshev_destroy and lobpcg_release_scratch return the rest.  The driver
// orders reuse by stream, so threads and streams may share the pool.
#include <mutex>

#include "kernels.cuh"

namespace lob {
namespace {

constexpr uint64_t kKeep = 64ull << 20;
constexpr int kDevices = 64;
std::mutex g_mutex;
cudaMemPool_t g_pool[kDevices] = {};
bool g_tried[kDevices] = {};

// the current device's pool, or null (then the default pool serves)
cudaMemPool_t pool_of_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_mutex);
  if (!g_tried[dev]) {
    g_tried[dev] = true;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    uint64_t keep = kKeep;
    if (cudaMemPoolCreate(&p, &props) == cudaSuccess &&
        cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess)
      g_pool[dev] = p;
    else
      cudaGetLastError();
  }
  return g_pool[dev];
}

}  // namespace

int scratch_alloc(void** p, size_t bytes, cudaStream_t st) {
  *p = nullptr;
  // a captured allocation belongs to the graph, whatever the pool, and making a
  // pool is no part of a capture
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) cudaGetLastError();
  cudaMemPool_t pool = cap == cudaStreamCaptureStatusNone ? pool_of_device() : nullptr;
  const size_t b = bytes < 16 ? 16 : bytes;
  if ((pool ? cudaMallocFromPoolAsync(p, b, pool, st) : cudaMallocAsync(p, b, st)) != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return LOBPCG_ERR_OOM;
  }
  return LOBPCG_OK;
}

void scratch_free(void* p, cudaStream_t st) {
  if (p) cudaFreeAsync(p, st);
}

// Memory whose free is still pending on a stream is not returned: callers have
// synchronised (cudaFree does, over the whole device).
void scratch_trim(int device) {
  if (device < 0 || device >= kDevices) return;
  std::lock_guard<std::mutex> lock(g_mutex);
  if (g_pool[device]) cudaMemPoolTrimTo(g_pool[device], 0);
}

}  // namespace lob

LOBPCG_EXPORT int lobpcg_release_scratch(void) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess)
    return LOBPCG_ERR_CUDA;
  lob::scratch_trim(dev);
  return LOBPCG_OK;
}
