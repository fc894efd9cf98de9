// Device memory of the library's objects and temporaries: one stream-ordered pool per device.
//
// cudaMalloc and cudaFree cost 35 to 150 us a call (and pinned allocations 120), so setting up a
// new pattern (two plans and a transpose, 26 device allocations at R-MAT scale 20) spent 1.1 of
// its 1.88 ms in them; from the pool a block costs 1 us, and the set-up 0.76 ms.  The pool keeps at
// most kPoolKeep bytes that no object uses: what is above that goes back to the driver at the next
// synchronisation, all of it when an allocation of the library fails, and the rest when the process
// ends.
#include <mutex>
#include <unordered_map>

#include "merbit_internal.cuh"

namespace merbit {

namespace {

constexpr unsigned long long kPoolKeep = 1ull << 30;

// The current device's pool, or null where it has none.
cudaMemPool_t pool_of(int dev) {
  static std::mutex mu;
  static std::unordered_map<int, cudaMemPool_t> pools;
  std::lock_guard<std::mutex> lock(mu);
  auto it = pools.find(dev);
  if (it != pools.end()) return it->second;
  // a small block that stays: device_wait's share its 2 MB of the address space, which would
  // be mapped and unmapped for each otherwise (65 us, 5 us with it)
  const RelaxedCalls relaxed;
  void* stays = nullptr;
  cudaMalloc(&stays, 256);
  cudaMemPool_t pool = nullptr;
  int ok = 0;
  if (cudaDeviceGetAttribute(&ok, cudaDevAttrMemoryPoolsSupported, dev) == cudaSuccess && ok) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    unsigned long long keep = kPoolKeep;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) pool = nullptr;
    else cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
  }
  cudaGetLastError();
  pools[dev] = pool;
  return pool;
}

// A refused allocation is the caller's answer, not an error of the next launch: the runtime would
// report it again there.
cudaError_t answered(cudaError_t e) {
  if (e == cudaErrorMemoryAllocation) cudaGetLastError();
  return e;
}

}  // namespace

// The block may be used by work queued on `st` from here on, and by any stream once `st` has been
// synchronised.  cudaFree does not wait for work that still uses a block of the pool: blocks that
// any stream may be using go through dev_free.  A stream that is being captured gets cudaMalloc (and its
// refusal): a pool allocation would become part of the graph.
cudaError_t dev_alloc(void** p, size_t bytes, cudaStream_t st) {
  *p = nullptr;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  const bool plain = cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone;
  cudaMemPool_t pool = plain ? nullptr : pool_of(dev);
  if (pool) {
    if (cudaMallocFromPoolAsync(p, bytes ? bytes : 1, pool, st) == cudaSuccess) return cudaSuccess;
    cudaGetLastError();
    cudaStreamSynchronize(st);
    cudaMemPoolTrimTo(pool, 0);
  }
  return answered(cudaMalloc(p, bytes ? bytes : 1));
}

cudaError_t dev_malloc(void** p, size_t bytes) {
  const cudaError_t e = answered(cudaMalloc(p, bytes));
  if (e != cudaErrorMemoryAllocation) return e;
  int dev = 0;
  cudaGetDevice(&dev);
  const cudaMemPool_t pool = pool_of(dev);
  if (!pool) return e;
  cudaMemPoolTrimTo(pool, 0);
  return answered(cudaMalloc(p, bytes));
}

cudaError_t device_wait(int device) {
  int current = device;
  cudaGetDevice(&current);
  if (current != device) cudaSetDevice(device);
  // cudaFree of a cudaMalloc block waits for the device.  cudaDeviceSynchronize does not where a
  // stream of any thread is being captured: it fails and breaks the capture.
  const RelaxedCalls relaxed;
  void* block = nullptr;
  cudaError_t e = answered(cudaMalloc(&block, 256));
  e = e == cudaSuccess ? cudaFree(block) : cudaDeviceSynchronize();
  if (current != device) cudaSetDevice(current);
  return e;
}

// Objects are destroyed from any thread, with any device current (a finaliser, say): the wait is
// for the device that holds the blocks.  Blocks that could not be waited for are left allocated
// rather than handed out again under running work.
void dev_free(int device, std::initializer_list<void*> blocks) {
  if (device_wait(device) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  const RelaxedCalls relaxed;
  for (void* b : blocks)
    if (b) cudaFree(b);
}

}  // namespace merbit
