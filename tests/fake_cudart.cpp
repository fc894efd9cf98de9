// A CUDA runtime without a GPU, for the host side of the library: device memory is host memory,
// launches do nothing, and the calls that allocate, free and wait keep to the runtime's rules
// (two devices):
//   * cudaFree of a cudaMalloc block waits for its device, of a pool block it does not: freeing a
//     pool block of a device that has work in flight is counted as a violation;
//   * cudaDeviceSynchronize waits for the current device; while a stream is being captured it
//     fails and breaks the capture;
//   * cudaMalloc and cudaFree break a global-mode capture unless the thread is in relaxed mode;
//   * idle memory of a pool counts against the device's memory until the pool is trimmed;
//   * a refused allocation is the next cudaGetLastError's answer too.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>

namespace {
struct Block { int dev; size_t bytes; bool pool; };
std::map<void*, Block> g_blocks;
int g_dev = 0, g_busy[2] = {0, 0}, g_violations = 0, g_capturing = 0, g_broken = 0, g_mallocs = 0;
cudaStreamCaptureMode g_mode = cudaStreamCaptureModeGlobal;
void* g_set = nullptr;      // the first range cleared since fake_reset
size_t g_set_bytes = 0;
cudaError_t g_last = cudaSuccess;
size_t g_used = 0, g_idle = 0, g_limit = ~size_t(0) >> 1;

cudaError_t unsafe_call() {
  if (!g_capturing || g_mode == cudaStreamCaptureModeRelaxed) return cudaSuccess;
  g_broken = 1;
  return cudaErrorStreamCaptureUnsupported;
}
cudaError_t take(void** p, size_t n, bool pool) {
  *p = std::calloc(1, n ? n : 1);
  g_blocks[*p] = Block{g_dev, n, pool};
  g_used += n;
  return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_reset() {
  g_dev = g_busy[0] = g_busy[1] = g_violations = g_capturing = g_broken = g_mallocs = 0;
  g_mode = cudaStreamCaptureModeGlobal;
  g_limit = ~size_t(0) >> 1;
  g_idle = 0;
  g_set = nullptr;
  g_last = cudaSuccess;
}
void fake_busy(int dev, int busy) { g_busy[dev] = busy; }
void fake_capture(int on) { g_capturing = on; }
void fake_limit(size_t more) { g_limit = g_used + g_idle + more; }
int fake_violations() { return g_violations; }
int fake_broken() { return g_broken; }
int fake_mallocs() { return g_mallocs; }
int fake_device() { return g_dev; }
void* fake_first_set(size_t* bytes) { *bytes = g_set_bytes; return g_set; }
size_t fake_used() { return g_used; }
size_t fake_idle() { return g_idle; }

cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_dev = d; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() {
  if (g_capturing) {
    g_broken = 1;
    return cudaErrorStreamCaptureUnsupported;
  }
  g_busy[g_dev] = 0;
  return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode* m) {
  const cudaStreamCaptureMode old = g_mode;
  g_mode = *m;
  *m = old;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = nullptr;
  if (cudaError_t e = unsafe_call()) return e;
  if (g_used + g_idle + n > g_limit) return g_last = cudaErrorMemoryAllocation;
  ++g_mallocs;
  return take(p, n, false);
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) {
  *p = nullptr;
  const size_t reuse = n < g_idle ? n : g_idle;
  if (g_used + g_idle + n - reuse > g_limit) return g_last = cudaErrorMemoryAllocation;
  g_idle -= reuse;
  return take(p, n, true);
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  if (cudaError_t e = unsafe_call()) return e;
  const auto it = g_blocks.find(p);
  if (it == g_blocks.end()) return cudaErrorInvalidValue;
  const Block b = it->second;
  if (!b.pool) g_busy[b.dev] = 0;
  else if (g_busy[b.dev]) ++g_violations;
  g_used -= b.bytes;
  if (b.pool) g_idle += b.bytes;
  std::free(p);
  g_blocks.erase(it);
  return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { g_idle = 0; return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { *p = (cudaMemPool_t)1; return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  if (!g_set) g_set = d, g_set_bytes = n;
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams* params) {
  static cudaGraph_t body[1];
  if (params->type == cudaGraphNodeTypeConditional) params->conditional.phGraph_out = body;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 4 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 227 << 10
       : a == cudaDevAttrMaxSharedMemoryPerMultiprocessor ? 228 << 10 : 1;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 2; return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) { std::memset(a, 0, sizeof *a); return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
  *c = s && g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
}
