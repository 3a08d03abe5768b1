// A stand-in for the CUDA runtime, for tests of the library's host side without
// a GPU: allocations are host memory that ends at an inaccessible page (a write
// or copy past an allocation's end is a SIGSEGV), copies and memsets happen at
// once, and kernels are only written to a log, which a test reads back.  A
// launch can be made to fail with fake_fail_launch().
#include <cuda_runtime.h>
#include <string.h>
#include <sys/mman.h>
#include <unistd.h>

#include <map>
#include <mutex>
#include <string>

namespace {

std::mutex g_mu;
std::string g_log;
std::map<const void*, std::string> g_names;        // host stub -> kernel name
struct Block { void* map; size_t len, bytes; bool host; };
std::map<uintptr_t, Block> g_blocks;
cudaError_t g_last = cudaSuccess;  // what cudaGetLastError returns next
long g_fail_alloc = 0;   // fails the n-th device allocation from now on (1-based); 0: none
long g_fail_launch = 0;  // fails the n-th launch from now on (1-based); 0: none
float g_ms = 1.f;

void note(const std::string& line) {
  std::lock_guard<std::mutex> lk(g_mu);
  g_log += line + "\n";
}

cudaError_t alloc(void** p, size_t bytes, bool host) {
  const size_t page = (size_t)sysconf(_SC_PAGESIZE), room = (bytes + page - 1) / page * page;
  char* m = (char*)mmap(nullptr, room + page, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (m == MAP_FAILED) return cudaErrorMemoryAllocation;
  mprotect(m + room, page, PROT_NONE);
  *p = m + (room - bytes) / 4 * 4;  // (ends within 3 bytes of the guard)
  std::lock_guard<std::mutex> lk(g_mu);
  g_blocks[(uintptr_t)*p] = Block{m, room + page, bytes, host};
  return cudaSuccess;
}

cudaError_t release(void* p) {
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_blocks.find((uintptr_t)p);
  if (it == g_blocks.end()) return p ? cudaErrorInvalidValue : cudaSuccess;
  munmap(it->second.map, it->second.len);
  g_blocks.erase(it);
  return cudaSuccess;
}

cudaError_t launched(const void* fn) {
  std::string name;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    name = g_names[fn];
    if (g_fail_launch > 0 && --g_fail_launch == 0) {
      g_log += "failed " + name + "\n";
      return g_last = cudaErrorLaunchOutOfResources;
    }
    g_log += "launch " + name + "\n";
  }
  return cudaSuccess;
}

std::string hex(const void* p) {
  char s[32];
  snprintf(s, sizeof(s), "%p", p);
  return s;
}

}  // namespace

extern "C" {

// ---- the test's side
const char* fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }
void fake_fail_launch(long n) { g_fail_launch = n; }
void fake_fail_alloc(long n) { g_fail_alloc = n; }

// ---- the runtime
cudaError_t cudaMalloc(void** p, size_t n) {
  if (g_fail_alloc > 0 && --g_fail_alloc == 0) return g_last = cudaErrorMemoryAllocation;
  return alloc(p, n, false);
}
cudaError_t cudaMallocHost(void** p, size_t n) { return alloc(p, n, true); }
cudaError_t cudaFree(void* p) { return release(p); }
cudaError_t cudaFreeHost(void* p) { return release(p); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  note("copy " + std::to_string((int)k) + " " + std::to_string(n));
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  note("memset " + hex(p) + " " + std::to_string(n));
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrClockRate ? 2070000 : 1;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "injected"; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = const_cast<void*>(s); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  std::lock_guard<std::mutex> lk(g_mu);
  memset(a, 0, sizeof(*a));
  auto it = g_blocks.upper_bound((uintptr_t)p);
  if (it == g_blocks.begin()) return cudaSuccess;
  --it;
  if ((uintptr_t)p >= it->first + it->second.bytes) return cudaSuccess;
  a->type = it->second.host ? cudaMemoryTypeHost : cudaMemoryTypeDevice;
  a->devicePointer = a->hostPointer = const_cast<void*>(p);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t) new char; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { delete (char*)s; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t) new char; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { delete (char*)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = g_ms; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) { *n = 4; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 4;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* fn, void**) { return launched(fn); }
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { *g = (cudaGraph_t) new char; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete (char*)g; return cudaSuccess; }
cudaError_t cudaGraphAddKernelNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t,
                                   const cudaKernelNodeParams* p) {
  *n = nullptr;
  note("node " + g_names[p->func]);
  return cudaSuccess;
}
cudaError_t cudaGraphKernelNodeSetAttribute(cudaGraphNode_t, cudaKernelNodeAttrID, const cudaKernelNodeAttrValue*) {
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = (cudaGraphExec_t) new char;
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { delete (char*)e; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { note("graph"); return cudaSuccess; }

// ---- what nvcc's host code calls
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
  g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(void** k, const void* fn) { *k = const_cast<void*>(fn); return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void* k, dim3, dim3, void**, size_t, cudaStream_t) { return launched(k); }

}  // extern "C"
