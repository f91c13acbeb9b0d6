// host_runtime.cpp -- a stand-in for the CUDA runtime, for tests of the library's host code on a
// machine without a GPU (tests/hostlib.py links it with the library's own objects).  Device memory is
// host memory with a settable limit, copies are done at once, kernels are recorded and not run.  An
// allocation can be made to fail, and a stream can be declared capturing: copies are then also recorded,
// as a graph would replay them.
#include <cuda_runtime.h>
#include <malloc.h>
#include <sys/mman.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <string>
#include <vector>

namespace {
struct Launch { std::string name; dim3 grid; };
struct Copy { const void* src; size_t bytes; std::string content; };
struct Owned { void* p; cudaHostFn_t destroy; };
std::map<const void*, std::string> kernels;
std::map<char*, size_t> blocks;  // live device allocations
std::vector<Launch> launches;
std::vector<Copy> copies;
std::vector<Owned> owned;  // what the captured graph keeps
size_t used = 0, peak = 0, limit = (size_t)256 << 30;
long long fail_in = 0, launch_fail_in = 0;  // the fail_in-th allocation (launch) from now fails
bool capturing = false;
cudaError_t last = cudaSuccess;
struct Config { dim3 grid, block; size_t smem; cudaStream_t st; };
thread_local std::vector<Config> configs;

cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) last = e;
  return e;
}
int encode_tensor_map(...) { return 0; }
}  // namespace

// ---- what a test sets and reads
extern "C" {
void host_limit(size_t bytes) { limit = bytes; }
void host_fail_in(long long n) { fail_in = n; }
void host_launch_fail_in(long long n) { launch_fail_in = n; }
void host_capture(int on) { capturing = on != 0; }
size_t host_used() { return used; }
size_t host_peak() { return peak; }
void host_clear() { launches.clear(); copies.clear(); peak = used; }
int host_launches() { return (int)launches.size(); }
const char* host_launch_name(int i) { return launches[i].name.c_str(); }
void host_launch_grid(int i, unsigned* g) { g[0] = launches[i].grid.x; g[1] = launches[i].grid.y; g[2] = launches[i].grid.z; }
// Recorded copies whose source no longer holds what it held when the copy was recorded.
int host_stale_copies() {
  int n = 0;
  for (auto& c : copies) n += memcmp(c.src, c.content.data(), c.bytes) != 0;
  return n;
}
int host_copies() { return (int)copies.size(); }
// Ends the captured graph's life; returns how many objects it kept.
int host_drop_graph() {
  for (auto& o : owned) o.destroy(o.p);
  const int n = (int)owned.size();
  owned.clear();
  return n;
}
}

// Freed host memory is overwritten, so that a copy recorded from it shows.
void operator delete(void* p) noexcept {
  if (p) memset(p, 0xDD, malloc_usable_size(p));
  free(p);
}
void operator delete(void* p, size_t) noexcept { operator delete(p); }
void* operator new(size_t n) {
  void* p = malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}

// ---- the runtime
extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  kernels[host] = name;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) {
  *k = (cudaKernel_t)host;
  return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, CUstream_st* st) {
  configs.push_back({grid, block, smem, st});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* st) {
  const Config c = configs.back();
  configs.pop_back();
  *grid = c.grid;
  *block = c.block;
  *smem = c.smem;
  *(cudaStream_t*)st = c.st;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t, cudaStream_t) {
  const bool ok = grid.x && grid.y && grid.z && grid.x < 0x80000000u && grid.y < 65536 && grid.z < 65536 && block.x &&
                  block.x * block.y * block.z <= 1024;
  if (!ok) return set(cudaErrorInvalidConfiguration);
  if (launch_fail_in > 0 && --launch_fail_in == 0) return set(cudaErrorLaunchOutOfResources);
  launches.push_back({kernels[(const void*)k], grid});
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* f, dim3 grid, dim3 block, void** a, size_t smem, cudaStream_t st) {
  return __cudaLaunchKernel((cudaKernel_t)f, grid, block, a, smem, st);
}

cudaError_t cudaMalloc(void** p, size_t n) {
  *p = nullptr;
  if ((fail_in > 0 && --fail_in == 0) || n > limit || used > limit - n) return set(cudaErrorMemoryAllocation);
  char* q = (char*)mmap(nullptr, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (q == (char*)MAP_FAILED) return set(cudaErrorMemoryAllocation);
  blocks[q] = n;
  used += n;
  if (used > peak) peak = used;
  *p = q;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  auto it = blocks.find((char*)p);
  if (it == blocks.end()) return p ? set(cudaErrorInvalidValue) : cudaSuccess;
  used -= it->second;
  munmap(p, it->second ? it->second : 1);
  blocks.erase(it);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (capturing) copies.push_back({s, n, std::string((const char*)s, n)});
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t) {
  for (size_t y = 0; y < h; ++y) memcpy((char*)d + y * dp, (const char*)s + y * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152
       : a == cudaDevAttrMaxSharedMemoryPerMultiprocessor ? 233472
       : a == cudaDevAttrReservedSharedMemoryPerBlock ? 1024
       : a == cudaDevAttrMaxRegistersPerMultiprocessor ? 65536
       : a == cudaDevAttrMaxThreadsPerMultiProcessor ? 2048
                                                           : 0;
  return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) { memset(p, 0, sizeof(*p)); return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  memset(a, 0, sizeof(*a));
  a->numRegs = 128;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = const_cast<void*>(s); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  memset(a, 0, sizeof(*a));
  a->type = cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = (void*)encode_tensor_map;
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)1; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, cudaStreamCaptureStatus* s, unsigned long long*, cudaGraph_t* g,
                                     const cudaGraphNode_t**, const cudaGraphEdgeData**, size_t*) {
  *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  if (g) *g = nullptr;
  return cudaSuccess;
}
cudaError_t cudaUserObjectCreate(cudaUserObject_t* o, void* p, cudaHostFn_t destroy, unsigned, unsigned) {
  owned.push_back({p, destroy});
  *o = nullptr;
  return cudaSuccess;
}
cudaError_t cudaGraphRetainUserObject(cudaGraph_t, cudaUserObject_t, unsigned, unsigned) { return cudaSuccess; }
cudaError_t cudaUserObjectRelease(cudaUserObject_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = nullptr; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
}
