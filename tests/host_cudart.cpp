// A CUDA runtime without a device, for tests of the library's host code: memory
// is the host's, copies and sets are done at once, kernels are noted by name and
// not run.  Allocations above a limit fail, and copies to the device from a given
// one on.  Loaded before libbern.so with its symbols global, so that the library's
// calls land here (tests/host_runtime.py).
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

struct Dim3 { unsigned x, y, z; };

namespace {
size_t alloc_limit = (size_t)-1;
long copies_left = -1;               // -1: all copies succeed
int copies = 0;
int last_error = 0;
std::map<const void*, std::string> names;
std::string launched;                // one name per line
std::string allocated;               // sizes in bytes, one per line
constexpr int kNoMemory = 2, kUnknown = 999;
int fail(int e) { return last_error = e; }
}  // namespace

extern "C" {
void host_set_alloc_limit(size_t bytes) { alloc_limit = bytes; }
void host_fail_copies_after(long n) { copies_left = n; }
int host_count_copies() { int n = copies; copies = 0; return n; }
const char* host_launched() { return launched.c_str(); }
const char* host_allocated() { return allocated.c_str(); }
void host_clear() { launched.clear(), allocated.clear(); }

int cudaMalloc(void** p, size_t n) {
  *p = nullptr;
  if (n > alloc_limit || !(*p = std::calloc(n ? n : 1, 1))) return fail(kNoMemory);
  allocated += std::to_string(n) + "\n";
  return 0;
}
int cudaFree(void* p) { std::free(p); return 0; }
int cudaMemGetInfo(size_t* f, size_t* t) { *f = *t = (size_t)1 << 30; return 0; }
int cudaMemcpy(void* d, const void* s, size_t n, int) {
  if (copies_left == 0) return fail(kUnknown);
  if (copies_left > 0) --copies_left;
  ++copies;
  std::memcpy(d, s, n);
  return 0;
}
int cudaMemcpyAsync(void* d, const void* s, size_t n, int k, void*) { return cudaMemcpy(d, s, n, k); }
int cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return 0; }
int cudaMemsetAsync(void* d, int v, size_t n, void*) { return cudaMemset(d, v, n); }
int cudaGetLastError() { int e = last_error; last_error = 0; return e; }
int cudaSetDevice(int) { return 0; }
int cudaGetDevice(int* d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int* v, int, int) { *v = 152; return 0; }
int cudaFuncSetAttribute(const void*, int, int) { return 0; }
int cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)s; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return 0;
}
int cudaStreamCreateWithFlags(void** s, unsigned) { *s = std::malloc(1); return 0; }
int cudaStreamDestroy(void* s) { std::free(s); return 0; }
int cudaStreamSynchronize(void*) { return 0; }
int cudaStreamWaitEvent(void*, void*, unsigned) { return 0; }
int cudaStreamIsCapturing(void*, int* s) { *s = 0; return 0; }
int cudaStreamBeginCapture(void*, int) { return 0; }
int cudaStreamEndCapture(void*, void** g) { *g = std::malloc(1); return 0; }
int cudaEventCreate(void** e) { *e = std::malloc(1); return 0; }
int cudaEventCreateWithFlags(void** e, unsigned) { *e = std::malloc(1); return 0; }
int cudaEventDestroy(void* e) { std::free(e); return 0; }
int cudaEventRecord(void*, void*) { return 0; }
int cudaEventSynchronize(void*) { return 0; }
int cudaEventElapsedTime(float* ms, void*, void*) { *ms = 1.0f; return 0; }
int cudaGraphInstantiate(void** x, void*, unsigned long long) { *x = std::malloc(1); return 0; }
int cudaGraphDestroy(void* g) { std::free(g); return 0; }
int cudaGraphExecDestroy(void* x) { std::free(x); return 0; }
int cudaGraphLaunch(void*, void*) { return 0; }

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*,
                            void*, void*, int*) {
  names[host] = name;
}
unsigned __cudaPushCallConfiguration(Dim3, Dim3, size_t, void*) { return 0; }
int __cudaPopCallConfiguration(Dim3* g, Dim3* b, size_t* s, void** st) {
  *g = *b = Dim3{1, 1, 1};
  *s = 0;
  *st = nullptr;
  return 0;
}
int __cudaGetKernel(void** k, const void* f) { *k = (void*)f; return 0; }
int __cudaLaunchKernel(void* k, Dim3, Dim3, void**, size_t, void*) {
  launched += names[k] + "\n";
  return 0;
}
}
