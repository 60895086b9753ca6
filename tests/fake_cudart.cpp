// A CUDA runtime without a GPU, for tests of the library's host code: linked with
// the library's own objects in place of the real runtime.  Device memory is host
// memory that nobody reads, copies and synchronisations do nothing, and launches
// are recorded by kernel name.  fake_fail_malloc(k) makes the k-th allocation from
// now on fail (and only that one), as a full device would.
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

namespace {
constexpr int kNoMemory = 2;  // cudaErrorMemoryAllocation
std::map<const void*, std::string> kernels;
std::vector<std::string> launched;
std::set<void*> live;
long fail_at = 0, mallocs = 0;
int last_error = 0;
int fake_encode() { return 0; }  // cuTensorMapEncodeTiled and the like: success
int fake_ctx(void** ctx) {
  static int c;
  *ctx = &c;
  return 0;
}
int launch(const void* f) {
  launched.push_back(kernels[f]);
  return 0;
}
int alloc(void** p, size_t n) {
  if (++mallocs == fail_at) {
    *p = nullptr;
    return last_error = kNoMemory;
  }
  *p = std::aligned_alloc(256, (n + 255) / 256 * 256 + 256);
  live.insert(*p);
  return 0;
}
int release(void* p) {
  if (p && !live.erase(p)) return last_error = 1;  // not ours, or freed twice
  std::free(p);
  return 0;
}
}  // namespace

struct Dim3 {
  unsigned x, y, z;
};

extern "C" {
// ---- what the tests ask
void fake_fail_malloc(long k) { mallocs = 0, fail_at = k; }
long fake_live() { return (long)live.size(); }
long fake_mallocs() { return mallocs; }
void fake_clear_launches() { launched.clear(); }
int fake_launches() { return (int)launched.size(); }
const char* fake_launch_name(int k) { return launched[k].c_str(); }

// ---- kernels
void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
  kernels[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(Dim3, Dim3, size_t, void*) { return 0; }
int __cudaPopCallConfiguration(Dim3* g, Dim3* b, size_t* smem, void* stream) {
  *g = *b = {1, 1, 1};
  *smem = 0;
  *static_cast<void**>(stream) = nullptr;
  return 0;
}
int __cudaGetKernel(const void** k, const void* host) {
  *k = host;
  return 0;
}
int __cudaLaunchKernel(const void* k, Dim3, Dim3, void**, size_t, void*) { return launch(k); }
int cudaLaunchKernel(const void* k, Dim3, Dim3, void**, size_t, void*) { return launch(k); }
int cudaFuncSetAttribute(const void*, int, int) { return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  *n = 1;
  return 0;
}

// ---- memory
int cudaMalloc(void** p, size_t n) { return alloc(p, n); }
int cudaMallocAsync(void** p, size_t n, void*) { return alloc(p, n); }
int cudaFree(void* p) { return release(p); }
int cudaFreeAsync(void* p, void*) { return release(p); }
int cudaMemcpy(void*, const void*, size_t, int) { return 0; }
int cudaMemcpyAsync(void*, const void*, size_t, int, void*) { return 0; }
int cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, int, void*) { return 0; }
int cudaMemset(void*, int, size_t) { return 0; }
int cudaMemsetAsync(void*, int, size_t, void*) { return 0; }
int cudaMemset2DAsync(void*, size_t, int, size_t, size_t, void*) { return 0; }
int cudaGetSymbolAddress(void** p, const void* s) {
  *p = const_cast<void*>(s);
  return 0;
}

// ---- device, streams, events, graphs
int cudaGetDevice(int* d) {
  *d = 0;
  return 0;
}
int cudaSetDevice(int) { return 0; }
int cudaDeviceSynchronize() { return 0; }
int cudaDeviceGetAttribute(int* v, int, int) {
  *v = 152;
  return 0;
}
int cudaGetDeviceProperties(void* prop, int) {
  std::strcpy(static_cast<char*>(prop), "fake");
  return 0;
}
int cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long, int* found) {
  *f = std::strcmp(name, "cuCtxGetCurrent") == 0 ? reinterpret_cast<void*>(fake_ctx)
                                                 : reinterpret_cast<void*>(fake_encode);
  if (found) *found = 0;
  return 0;
}
int cudaGetLastError() {
  const int e = last_error;
  last_error = 0;
  return e;
}
const char* cudaGetErrorName(int) { return "fake"; }
const char* cudaGetErrorString(int) { return "fake"; }
static int handle(void** h) {
  static char c;
  *h = &c;
  return 0;
}
int cudaStreamCreateWithFlags(void** s, unsigned) { return handle(s); }
int cudaStreamDestroy(void*) { return 0; }
int cudaStreamSynchronize(void*) { return 0; }
int cudaStreamWaitEvent(void*, void*, unsigned) { return 0; }
int cudaStreamBeginCapture(void*, int) { return 0; }
int cudaStreamEndCapture(void*, void** g) { return handle(g); }
int cudaEventCreate(void** e) { return handle(e); }
int cudaEventCreateWithFlags(void** e, unsigned) { return handle(e); }
int cudaEventDestroy(void*) { return 0; }
int cudaEventRecord(void*, void*) { return 0; }
int cudaEventSynchronize(void*) { return 0; }
int cudaEventElapsedTime(float* ms, void*, void*) {
  *ms = 1.0f;
  return 0;
}
int cudaGraphInstantiate(void** x, void*, unsigned long long) { return handle(x); }
int cudaGraphLaunch(void*, void*) { return 0; }
int cudaGraphDestroy(void*) { return 0; }
int cudaGraphExecDestroy(void*) { return 0; }
}
