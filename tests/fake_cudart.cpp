// A stand-in for the CUDA runtime, preloaded before libcudart by test_host_failures.py: device memory is host memory
// of a limited size, kernels do nothing but leave their names, copies are real and checked against the blocks they
// touch.  It gives the host code of the library the failures a GPU test must not provoke: an allocation that fails, a
// launch that fails, a stream under capture, a second device.
#include <cuda_runtime_api.h>
#include <sys/mman.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace {
struct Pool {
  int dev;
  size_t used = 0, reserved = 0;
  uint64_t keep = 0;  // release threshold
};
struct Block {
  size_t bytes;
  Pool* pool;  // null: cudaMalloc or pinned
  bool device;
};
std::mutex mu;
std::map<char*, Block> blocks;
std::map<const void*, std::string> names;
std::vector<std::string> launched;
std::vector<Pool*> pools;  // [0, kDevices) are the default pools
constexpr int kDevices = 2;
size_t memory = size_t(1) << 40, plain = 0, largest = 0;
int device = 0, launch_error = 0, capturing = 0, out_of_range = 0;
cudaError_t last = cudaSuccess;
struct Call {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
};
thread_local Call call;

Pool* default_pool(int d) {
  while ((int)pools.size() < kDevices) pools.push_back(new Pool{(int)pools.size()});
  return pools[d];
}
size_t held() {  // what no other allocation can have
  size_t t = plain;
  for (Pool* p : pools) t += p->reserved;
  return t;
}
cudaError_t fail(cudaError_t e) { return last = e; }
cudaError_t give(void** p, size_t n, Pool* pool, bool dev) {
  std::lock_guard<std::mutex> lk(mu);
  size_t more = !dev ? 0 : n;
  if (pool) more = pool->used + n > pool->reserved ? pool->used + n - pool->reserved : 0;
  if (held() + more > memory) {  // the driver takes back what pools do not use
    for (Pool* q : pools) q->reserved = q->used;
    if (pool) more = n;
    if (held() + more > memory) return fail(cudaErrorMemoryAllocation);
  }
  *p = mmap(nullptr, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (*p == MAP_FAILED) abort();
  blocks[(char*)*p] = Block{n, pool, dev};
  if (dev && n > largest) largest = n;
  if (pool) {
    pool->used += n;
    if (pool->used > pool->reserved) pool->reserved = pool->used;
  } else if (dev) {
    plain += n;
  }
  return cudaSuccess;
}
cudaError_t take(void* p) {
  std::lock_guard<std::mutex> lk(mu);
  auto it = blocks.find((char*)p);
  if (!p) return cudaSuccess;
  if (it == blocks.end()) return fail(cudaErrorInvalidValue);
  if (it->second.pool) it->second.pool->used -= it->second.bytes;
  else if (it->second.device) plain -= it->second.bytes;
  munmap(p, it->second.bytes ? it->second.bytes : 1);
  blocks.erase(it);
  return cudaSuccess;
}
void sync() {
  std::lock_guard<std::mutex> lk(mu);
  for (Pool* p : pools) p->reserved = std::max<size_t>(p->used, std::min<size_t>(p->reserved, p->keep));
}
bool inside(const void* p, size_t n) {  // ranges that start in a known block must end in it
  std::lock_guard<std::mutex> lk(mu);
  auto it = blocks.upper_bound((char*)p);
  if (it == blocks.begin()) return true;
  --it;
  const size_t at = (char*)p - it->first;
  if (at >= std::max<size_t>(it->second.bytes, 1) || at + n <= it->second.bytes) return true;
  ++out_of_range;
  return false;
}
}  // namespace

extern "C" {
void fake_memory_left(size_t n) {  // beyond what is in use
  memory = plain + n;
  for (Pool* p : pools) memory += p->used;
}
size_t fake_pool_kept() {
  size_t t = 0;
  for (Pool* p : pools) t += p->reserved - p->used;
  return t;
}
size_t fake_pool_kept_on(int d) {
  size_t t = 0;
  for (Pool* p : pools) t += p->dev == d ? p->reserved - p->used : 0;
  return t;
}
unsigned long long fake_default_threshold(int d) { return default_pool(d)->keep; }
size_t fake_largest() { size_t n = largest; largest = 0; return n; }
int fake_out_of_range() { return out_of_range; }
void fake_launch_error(int e) { launch_error = e; }
void fake_capturing(int on) { capturing = on; }
void fake_device(int d) { device = d; }
int fake_launches() { return (int)launched.size(); }
const char* fake_launched(int i) { return launched[i].c_str(); }
void fake_forget() { launched.clear(); }

cudaError_t cudaMalloc(void** p, size_t n) { return give(p, n, nullptr, true); }
cudaError_t cudaMallocHost(void** p, size_t n) { return give(p, n, nullptr, false); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return give(p, n, default_pool(device), true); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t pool, cudaStream_t) { return give(p, n, (Pool*)pool, true); }
cudaError_t cudaFree(void* p) { return take(p); }
cudaError_t cudaFreeHost(void* p) { return take(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return take(p); }
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* p, int d) { *p = (cudaMemPool_t)default_pool(d); return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps* props) {
  default_pool(0);
  pools.push_back(new Pool{props->location.id});
  *p = (cudaMemPool_t)pools.back();
  return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) {
  ((Pool*)p)->reserved = ((Pool*)p)->used;
  ((Pool*)p)->keep = 0;
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t p, cudaMemPoolAttr a, void* v) {
  if (a == cudaMemPoolAttrReleaseThreshold) ((Pool*)p)->keep = *(uint64_t*)v;
  return cudaSuccess;
}
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t p, cudaMemPoolAttr a, void* v) {
  if (a == cudaMemPoolAttrReleaseThreshold) *(uint64_t*)v = ((Pool*)p)->keep;
  return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t n) {
  Pool* q = (Pool*)p;
  q->reserved = std::max(q->used, std::min(q->reserved, n));
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (!inside(d, n) || !inside(s, n)) return fail(cudaErrorInvalidValue);
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  if (!inside(d, n)) return fail(cudaErrorInvalidValue);
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { device = d; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = kDevices; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { sync(); return cudaSuccess; }
cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "fake error"; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { static char block[1 << 8]; *p = block; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)malloc(8); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { sync(); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
  *c = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { capturing = 1; return cudaSuccess; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                                          cudaStreamCaptureMode) { capturing = 1; return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { capturing = 0; *g = (cudaGraph_t)&capturing; return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)malloc(8); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { *g = (cudaGraph_t)&capturing; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = (cudaGraphExec_t)&capturing; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned) { *h = 0; return cudaSuccess; }
cudaError_t cudaGraphAddNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams* p) {
  static cudaGraph_t body = (cudaGraph_t)&capturing;
  p->conditional.phGraph_out = &body;
  return cudaSuccess;
}

// what the compiler's launch stubs call
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t n, cudaStream_t s) { call = Call{g, b, n, s}; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* n, void* s) {
  *g = call.grid;
  *b = call.block;
  *n = call.smem;
  *(cudaStream_t*)s = call.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) { *k = (cudaKernel_t)host; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void**, size_t, cudaStream_t) {
  std::lock_guard<std::mutex> lk(mu);
  if (launch_error) return fail((cudaError_t)launch_error);
  launched.push_back(names[(const void*)k] + " " + std::to_string(g.x) + " " + std::to_string(g.y) + " " + std::to_string(g.z));
  return cudaSuccess;
}
}
