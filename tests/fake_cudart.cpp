// A stand-in for the CUDA runtime, preloaded in front of it: device memory is
// a range of addresses and a budget, kernels and copies do nothing, and every
// call is counted, so that what the library's host code allocates, frees and
// waits for can be tested without a GPU.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <map>
#include <mutex>
#include <set>
#include <string>

namespace {

struct Block {
  size_t bytes;
  bool ordered;  // from cudaMallocAsync
};

std::recursive_mutex mu;
std::map<std::string, int> calls;
std::map<void *, Block> device;
std::set<void *> pinned;
size_t total = (size_t)280 << 30, used = 0;
size_t reserved = 0;  // of `used`: freed in stream order, until a synchronisation or a trim
unsigned long long next_address = 1ull << 40;
unsigned node_threads = 0;  // most threads of a graph's kernel so far
bool capture_open = false;  // some stream of the device is being captured
thread_local cudaError_t last = cudaSuccess;

cudaError_t done(const char *name, cudaError_t e = cudaSuccess) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  ++calls[name];
  if (e != cudaSuccess) last = e;
  return e;
}

cudaError_t take(const char *name, void **p, size_t bytes, bool ordered) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  const size_t again = ordered && bytes < reserved ? bytes : ordered ? reserved : 0;
  if (bytes - again > total - used) return done(name, cudaErrorMemoryAllocation);
  reserved -= again;
  used += bytes - again;
  *p = reinterpret_cast<void *>(next_address);
  next_address += (bytes + 4095) / 4096 * 4096;
  device[*p] = {bytes, ordered};
  return done(name);
}

cudaError_t give(const char *name, void *p, bool stream_ordered) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  if (!p) return done(name);
  const auto it = device.find(p);
  if (it == device.end() || (stream_ordered && !it->second.ordered)) return done(name, cudaErrorInvalidValue);
  if (it->second.ordered) reserved += it->second.bytes;
  else used -= it->second.bytes;
  device.erase(it);
  return done(name);
}

void trim() {
  std::lock_guard<std::recursive_mutex> lk(mu);
  used -= reserved;
  reserved = 0;
}

// While a stream is captured, the device and the legacy stream cannot be synchronised.
cudaError_t sync(const char *name, bool refused) {
  if (!refused) trim();
  return done(name, refused ? cudaErrorStreamCaptureUnsupported : cudaSuccess);
}

cudaError_t kernel_node(const char *name, const cudaKernelNodeParams *p) {
  const unsigned threads = p->gridDim.x * p->blockDim.x;
  if (threads > node_threads) node_threads = threads;
  return done(name);
}

template <typename T>
cudaError_t handle(const char *name, T *out) {
  *out = reinterpret_cast<T>(std::malloc(1));
  return done(name);
}

cudaError_t drop(const char *name, void *h) {
  std::free(h);
  return done(name);
}

}  // namespace

extern "C" {

// ---- control
void fake_clear() {
  std::lock_guard<std::recursive_mutex> lk(mu);
  calls.clear();
}
int fake_calls(const char *name) {
  std::lock_guard<std::recursive_mutex> lk(mu);
  const auto it = calls.find(name);
  return it == calls.end() ? 0 : it->second;
}
void fake_capture(int open) { capture_open = open != 0; }
void fake_total(size_t bytes) { total = bytes; }
size_t fake_used() { return used; }
unsigned fake_node_threads() { return node_threads; }

// ---- device
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrL2CacheSize ? 129 << 20 : 1;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return sync(__func__, capture_open); }
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
cudaError_t cudaPeekAtLastError() { return last; }

// ---- memory
cudaError_t cudaMalloc(void **p, size_t bytes) { return take(__func__, p, bytes, false); }
cudaError_t cudaMallocAsync(void **p, size_t bytes, cudaStream_t) { return take(__func__, p, bytes, true); }
cudaError_t cudaFree(void *p) { return give(__func__, p, false); }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return give(__func__, p, true); }
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t *pool, int) {
  *pool = nullptr;
  return done(__func__);
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) {
  trim();
  return done(__func__);
}
cudaError_t cudaMallocHost(void **p, size_t bytes) {
  *p = std::calloc(1, bytes);
  pinned.insert(*p);
  return done(__func__);
}
cudaError_t cudaHostAlloc(void **p, size_t bytes, unsigned) { return cudaMallocHost(p, bytes); }
cudaError_t cudaFreeHost(void *p) {
  pinned.erase(p);
  std::free(p);
  return done(__func__);
}
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) {
  *d = h;
  return done(__func__);
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *p) {
  *a = {};
  a->type = pinned.count(const_cast<void *>(p)) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
  return done(__func__);
}
cudaError_t cudaMemcpy(void *, const void *, size_t, cudaMemcpyKind) { return done(__func__); }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return done(__func__); }
cudaError_t cudaMemcpyToSymbol(const void *, const void *, size_t, size_t, cudaMemcpyKind) { return done(__func__); }
cudaError_t cudaMemset(void *, int, size_t) { return done(__func__); }
cudaError_t cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return done(__func__); }

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return handle(__func__, s); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return drop(__func__, s); }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return sync(__func__, capture_open && !s); }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *st) {
  *st = cudaStreamCaptureStatusNone;
  return done(__func__);
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return done(__func__); }
cudaError_t cudaEventCreate(cudaEvent_t *e) { return handle(__func__, e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return handle(__func__, e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return drop(__func__, e); }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return done(__func__); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return done(__func__); }
cudaError_t cudaEventQuery(cudaEvent_t) { return done(__func__); }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return done(__func__);
}
cudaError_t cudaGraphCreate(cudaGraph_t *g, unsigned) { return handle(__func__, g); }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return drop(__func__, g); }
cudaError_t cudaGraphAddMemcpyNode1D(cudaGraphNode_t *n, cudaGraph_t, const cudaGraphNode_t *, size_t, void *,
                                     const void *, size_t, cudaMemcpyKind) {
  *n = nullptr;
  return done(__func__);
}
cudaError_t cudaGraphAddKernelNode(cudaGraphNode_t *n, cudaGraph_t, const cudaGraphNode_t *, size_t,
                                   const cudaKernelNodeParams *p) {
  *n = nullptr;
  return kernel_node(__func__, p);
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) { return handle(__func__, e); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { return drop(__func__, e); }
cudaError_t cudaGraphExecKernelNodeSetParams(cudaGraphExec_t, cudaGraphNode_t, const cudaKernelNodeParams *p) {
  return kernel_node(__func__, p);
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return done(__func__); }

// ---- kernels
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t) { return done(__func__); }
cudaError_t cudaLaunchCooperativeKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t) {
  return done(__func__);
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *) {
  *k = nullptr;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) {
  return done("cudaLaunchKernel");
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return done(__func__); }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
  *n = 1;
  return done(__func__);
}

}  // extern "C"
