// scratch.cu -- device scratch of the calls that work on host arrays (batch
// EOS, network inference, loss gradient and temperature guesses).
//
// These calls need device room for their arrays only while they run.  A
// cudaMalloc and a cudaFree per call took longer than the work itself on
// small batches (the network's inference and gradient over 65536 samples:
// ~280 of 450 us), so the room comes from a memory pool of the library's own,
// one per device, allocated and freed in stream order: calls from several
// threads and on several streams each get room of their own.  The pool keeps
// at most KEEP bytes between calls, and nothing once the last EOS table and
// network are destroyed.
#include <cuda_runtime.h>

#include <mutex>

#include "phl.h"
#include "phl_internal.cuh"

namespace phl {
namespace {

constexpr int MAX_DEV = 64;
constexpr unsigned long long KEEP = 256ull << 20;   // 3.5e6 batch-EOS states; larger calls give the rest back

std::mutex mu;
cudaMemPool_t pools[MAX_DEV] = {};
long owners = 0;

cudaError_t pool_of(int dev, cudaMemPool_t *out) {
  if (dev < 0 || dev >= MAX_DEV) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> l(mu);
  if (!pools[dev]) {
    cudaMemPoolProps p = {};
    p.allocType = cudaMemAllocationTypePinned;
    p.handleTypes = cudaMemHandleTypeNone;
    p.location.type = cudaMemLocationTypeDevice;
    p.location.id = dev;
    cudaMemPool_t q = nullptr;
    cudaError_t e = cudaMemPoolCreate(&q, &p);
    unsigned long long keep = KEEP;
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(q, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
      if (q) cudaMemPoolDestroy(q);
      return e;
    }
    pools[dev] = q;
  }
  *out = pools[dev];
  return cudaSuccess;
}

}  // namespace

cudaError_t CallScratch::get(size_t bytes, cudaStream_t stream) {
  // not under capture: the call copies to and from the host and waits
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(stream, &cap);
  if (e != cudaSuccess) return e;
  if (cap != cudaStreamCaptureStatusNone) return cudaErrorStreamCaptureUnsupported;
  int dev = 0;
  cudaMemPool_t pool = nullptr;
  e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = pool_of(dev, &pool);
  if (e == cudaSuccess) e = cudaMallocFromPoolAsync(&p, bytes, pool, stream);
  if (e != cudaSuccess) p = nullptr;
  s = stream;
  return e;
}

CallScratch::~CallScratch() {
  if (p) cudaFreeAsync(p, s);
}

void scratch_owner(int change) {
  std::lock_guard<std::mutex> l(mu);
  owners += change;
  if (owners > 0) return;
  int cur = 0;
  if (cudaGetDevice(&cur) != cudaSuccess) return;
  for (int d = 0; d < MAX_DEV; ++d)
    if (pools[d]) {
      cudaSetDevice(d);
      cudaDeviceSynchronize();   // a free that is still in stream order would keep its room
      cudaMemPoolTrimTo(pools[d], 0);
    }
  cudaSetDevice(cur);
}

}  // namespace phl
