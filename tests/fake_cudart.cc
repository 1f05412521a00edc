// A CUDA runtime that holds "device" memory on the host and runs no kernel, for
// tests of the library's host code without a GPU: what a handle and a plan
// allocate, and what is left after an allocation fails.  The library's objects are
// linked against this file instead of the CUDA runtime (test_host_memory_cpu.py).
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {
std::map<void*, size_t> blocks, pinned;
size_t live = 0, limit = (size_t)1 << 42;
long countdown = -1;                     // allocations left before one fails (-1: none does)
long pinned_calls = 0;
int last = 0;
// A clock for tests of what the library times: each launch advances it by the cost
// of its kernel, the sum over the set patterns that the mangled name contains.  With
// no cost set every interval is 1 ms.
std::map<const void*, std::string> kernels;
std::map<std::string, double> costs;
double now = 0.0;

int grab(std::map<void*, size_t>& m, void** p, size_t n) {
  *p = nullptr;
  if (countdown >= 0 && countdown-- == 0) { countdown = -1; return last = 2; }
  *p = std::calloc(n ? n : 1, 1);        // pages that nothing touches cost nothing
  m[*p] = n;
  return 0;
}
int drop(std::map<void*, size_t>& m, void* p) {
  if (!p) return 0;
  m.erase(p);
  std::free(p);
  return 0;
}
int encode(...) { return 0; }
struct Dim3 { unsigned x, y, z; };
}  // namespace

extern "C" {
// what the tests set and read
void fake_fail_after(long n) { countdown = n; }
size_t fake_device_bytes() { return live; }
size_t fake_pinned_blocks() { return pinned.size(); }
long fake_pinned_calls() { return pinned_calls; }
void fake_cost(const char* pattern, double ms) { costs[pattern] = ms; }

int cudaMalloc(void** p, size_t n) {
  if (live + n > limit) { *p = nullptr; return last = 2; }
  const int e = grab(blocks, p, n);
  if (!e) live += n;
  return e;
}
int cudaFree(void* p) {
  if (p) live -= blocks.at(p);
  return drop(blocks, p);
}
int cudaMallocAsync(void** p, size_t n, void*) { return cudaMalloc(p, n); }
int cudaFreeAsync(void* p, void*) { return cudaFree(p); }
int cudaMallocHost(void** p, size_t n) { ++pinned_calls; return grab(pinned, p, n); }
int cudaFreeHost(void* p) { return drop(pinned, p); }
int cudaMemGetInfo(size_t* f, size_t* t) { *f = limit - live; *t = limit; return 0; }
int cudaMemcpy(void* d, const void* s, size_t n, int) { std::memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int, void*) { std::memcpy(d, s, n); return 0; }
int cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, int, void*) {
  for (size_t i = 0; i < h; ++i) std::memcpy((char*)d + i * dp, (const char*)s + i * sp, w);
  return 0;
}
int cudaMemset(void* p, int v, size_t n) { std::memset(p, v, n); return 0; }
int cudaMemsetAsync(void* p, int v, size_t n, void*) { std::memset(p, v, n); return 0; }
int cudaGetLastError() { const int e = last; last = 0; return e; }
const char* cudaGetErrorString(int) { return "fake"; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaGetDeviceCount(int* n) { *n = 1; return 0; }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 152; return 0; }
int cudaFuncGetAttributes(void*, const void*) { return 1; }
int cudaFuncSetAttribute(const void*, int, int) { return 0; }
int cudaGetSymbolAddress(void**, const void*) { return 1; }
int cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long, int* q) {
  *f = (void*)encode;
  *q = 0;
  return 0;
}
int cudaEventCreate(void** e) { *e = new double(0.0); return 0; }
int cudaEventCreateWithFlags(void** e, unsigned) { return cudaEventCreate(e); }
int cudaEventDestroy(void* e) { delete static_cast<double*>(e); return 0; }
int cudaEventElapsedTime(float* ms, void* a, void* b) {
  *ms = costs.empty() ? 1.f : (float)(*static_cast<double*>(b) - *static_cast<double*>(a));
  return 0;
}
int cudaEventRecord(void* e, void*) { *static_cast<double*>(e) = now; return 0; }
int cudaEventRecordWithFlags(void*, void*, unsigned) { return 0; }
int cudaEventSynchronize(void*) { return 0; }
int cudaGraphDestroy(void*) { return 0; }
int cudaGraphExecDestroy(void*) { return 0; }
int cudaGraphInstantiate(void** g, void*, unsigned long long) { *g = &last; return 0; }
int cudaGraphLaunch(void*, void*) { return 0; }
int cudaStreamBeginCapture(void*, int) { return 0; }
int cudaStreamEndCapture(void*, void** g) { *g = &last; return 0; }
int cudaStreamCreateWithFlags(void** s, unsigned) { *s = &last; return 0; }
int cudaStreamDestroy(void*) { return 0; }
int cudaStreamIsCapturing(void*, int* c) { *c = 0; return 0; }
int cudaStreamSynchronize(void*) { return 0; }
int cudaLaunchKernelExC(const void*, const void*, void**) { return 0; }
int __cudaLaunchKernel(void* k, Dim3, Dim3, void**, size_t, void*) {
  for (const auto& c : costs) if (kernels[k].find(c.first) != std::string::npos) now += c.second;
  return 0;
}
int __cudaGetKernel(void** k, const void* f) { *k = const_cast<void*>(f); return 0; }
unsigned __cudaPushCallConfiguration(Dim3, Dim3, size_t, void*) { return 0; }
int __cudaPopCallConfiguration(void*, void*, size_t* n, void*) { *n = 0; return 0; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, void*, void*, void*, void*, int*) {
  kernels[f] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
