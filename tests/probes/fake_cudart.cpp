// A CUDA runtime without a device, for tests of the library's host code: every entry point that
// the library calls.  Kernels do nothing.  Work on a stream is done only when something waits for it
// (so the order in which the host code waits can be observed), device memory is host memory
// against a limit, and the calls that the tests look at are counted.
#include <cuda_runtime_api.h>

#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <string>
#include <vector>

namespace {

struct Dep;
struct Stream {
  unsigned long long enqueued = 0, done = 0;
  std::vector<Dep> deps;
};
struct Dep {
  unsigned long long at;  // operations of the stream after this one wait
  Stream* on;
  unsigned long long upto;
};
struct Event {
  Stream* s = nullptr;
  unsigned long long upto = 0;
};

std::map<cudaStream_t, Stream*> g_streams;
std::map<void*, size_t> g_mem;
std::vector<std::string> g_launched;
size_t g_limit = (size_t)280 << 30, g_used = 0, g_largest = ~(size_t)0, g_pool_kept = 0;
unsigned long long g_most_pending_at_free = 0;
unsigned g_trims = 0, g_copies = 0;
int g_host_blocks = 0, g_capturing = 0, g_events = 0, g_queries = 0;
int g_cluster_room = 1;
int g_pool_obj;  // the library's pool
cudaError_t g_last = cudaSuccess;

// kernels register before this file's own objects are made
std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> m;
  return m;
}

Stream* stream(cudaStream_t s) {
  Stream*& x = g_streams[s];
  if (!x) x = new Stream();
  return x;
}

void complete(Stream* s, unsigned long long upto) {
  if (s->done >= upto) return;
  s->done = upto;
  for (size_t k = 0; k < s->deps.size(); ++k)
    if (s->deps[k].at < upto) complete(s->deps[k].on, s->deps[k].upto);
}

void op(cudaStream_t s) { ++stream(s)->enqueued; }

unsigned long long pending() {
  unsigned long long n = 0;
  for (auto& x : g_streams) n += x.second->enqueued - x.second->done;
  return n;
}

cudaError_t fail(cudaError_t e) { return g_last = e; }

cudaError_t take(void** p, size_t bytes) {
  *p = nullptr;
  if (bytes > g_largest || g_used + bytes > g_limit) return fail(cudaErrorMemoryAllocation);
  *p = aligned_alloc(512, (bytes + 511) / 512 * 512);
  if (!*p) return fail(cudaErrorMemoryAllocation);
  if (bytes < ((size_t)64 << 20)) memset(*p, 0, bytes);
  g_mem[*p] = bytes;
  g_used += bytes;
  return cudaSuccess;
}

cudaError_t give(void* p) {
  if (!p) return cudaSuccess;
  g_most_pending_at_free = std::max(g_most_pending_at_free, pending());
  auto it = g_mem.find(p);
  if (it == g_mem.end()) return fail(cudaErrorInvalidValue);
  g_used -= it->second;
  g_mem.erase(it);
  free(p);
  return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- what the tests set and read ----
void fake_reset() {
  g_limit = (size_t)280 << 30;
  g_largest = ~(size_t)0;
  g_most_pending_at_free = 0;
  g_trims = g_copies = 0;
  g_capturing = 0;
  g_cluster_room = 1;
  g_launched.clear();
}
void fake_memory(size_t limit, size_t largest) { g_limit = g_used + limit, g_largest = largest; }
unsigned long long fake_used() { return g_used; }
unsigned long long fake_pending() { return pending(); }
unsigned long long fake_most_pending_at_free() { return g_most_pending_at_free; }
unsigned fake_trims() { return g_trims; }
unsigned fake_copies() { return g_copies; }
int fake_host_blocks() { return g_host_blocks; }
int fake_events() { return g_events; }
int fake_queries() { return g_queries; }
void fake_capturing(int on) { g_capturing = on; }
void fake_cluster_room(int clusters) { g_cluster_room = clusters; }
int fake_launched(const char* what) {
  int n = 0;
  for (auto& s : g_launched) n += s.find(what) != std::string::npos;
  return n;
}

// ---- registration and launches ----
void** __cudaRegisterFatBinary(void*) {
  static void* h[1];
  return h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 0; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names()[host] = name;
}
static dim3 g_grid, g_block;
static size_t g_smem;
static cudaStream_t g_on;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* s) {
  g_grid = grid, g_block = block, g_smem = smem, g_on = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
  *grid = g_grid, *block = g_block, *smem = g_smem, *(cudaStream_t*)s = g_on;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t s) {
  g_launched.push_back(names()[(const void*)k]);
  op(s);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  bool cluster = false;
  for (unsigned k = 0; k < c->numAttrs; ++k) cluster |= c->attrs[k].id == cudaLaunchAttributeClusterDimension;
  if (cluster && g_cluster_room == 0) return fail(cudaErrorInvalidClusterSize);
  g_launched.push_back((cluster ? "cluster:" : "") + names()[f]);
  op(c->stream);
  return cudaSuccess;
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void**, size_t, cudaStream_t s) {
  g_launched.push_back("cooperative:" + names()[f]);
  op(s);
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, enum cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = g_cluster_room;
  return cudaSuccess;
}

// ---- device ----
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "(fake runtime)"; }
cudaError_t cudaDeviceSynchronize() {
  for (auto& x : g_streams) complete(x.second, x.second->enqueued);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  *p = nullptr;
  return fail(cudaErrorInvalidSymbol);
}

// ---- memory ----
cudaError_t cudaMemGetInfo(size_t* fr, size_t* total) {
  *fr = g_limit > g_used ? g_limit - g_used : 0;
  *total = g_limit;
  return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const struct cudaMemPoolProps*) {
  *p = (cudaMemPool_t)&g_pool_obj;
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, enum cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t) {
  if (p == (cudaMemPool_t)&g_pool_obj) ++g_trims;
  return cudaSuccess;
}
cudaError_t cudaMallocAsync(void** p, size_t bytes, cudaStream_t) {
  return take(p, bytes);
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t bytes, cudaMemPool_t, cudaStream_t) {
  return take(p, bytes);
}
cudaError_t cudaFree(void* p) { return give(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t s) {
  auto it = g_mem.find(p);
  if (it == g_mem.end()) return fail(cudaErrorInvalidValue);
  op(s);
  g_used -= it->second;
  g_mem.erase(it);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned) {
  *p = calloc(1, bytes);
  g_host_blocks += *p != nullptr;
  return *p ? cudaSuccess : fail(cudaErrorMemoryAllocation);
}
cudaError_t cudaFreeHost(void* p) {
  g_host_blocks -= p != nullptr;
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* src, size_t n, enum cudaMemcpyKind, cudaStream_t s) {
  memcpy(d, src, n);
  ++g_copies;
  op(s);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t s) {
  op(s);
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof(*a));
  a->type = cudaMemoryTypeDevice;
  a->devicePointer = const_cast<void*>(p);
  return cudaSuccess;
}

// ---- streams and events ----
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t) new int(0);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  complete(stream(s), stream(s)->enqueued);
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, enum cudaStreamCaptureStatus* c) {
  *c = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(enum cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  *e = (cudaEvent_t) new Event();
  ++g_events;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  delete (Event*)e;
  --g_events;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  ((Event*)e)->s = stream(s);
  ((Event*)e)->upto = stream(s)->enqueued;
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t e) {
  if (((Event*)e)->s) complete(((Event*)e)->s, ((Event*)e)->upto);
  return cudaSuccess;
}
cudaError_t cudaEventQuery(cudaEvent_t e) {
  Event* v = (Event*)e;
  ++g_queries;
  return !v->s || v->s->done >= v->upto ? cudaSuccess : cudaErrorNotReady;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.0f;
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  Event* v = (Event*)e;
  if (v->s) stream(s)->deps.push_back(Dep{stream(s)->enqueued, v->s, v->upto});
  return cudaSuccess;
}

}  // extern "C"
