// A CUDA runtime without a GPU, for tests of the library's host side: the
// library's object files are linked against these functions instead of the
// runtime (tests/fake_cuda.py).  Device memory is host memory, a launch checks
// its grid and is logged and not run, an allocation can be made to fail, and
// the current device is a number the test sets.  Copies and fills up to 1 MB
// are carried out, larger ones not.
#include <cuda_runtime_api.h>
#include <cxxabi.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

static std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> m;
  return m;
}
static std::vector<std::string> g_log;
static std::map<void*, size_t> g_mem;
static size_t g_live = 0, g_peak = 0;
static int g_device = 0;
static long g_fail = 0, g_allocs = 0;
static cudaError_t g_last = cudaSuccess;

static std::string demangled(const void* f) {
  const std::string& n = names()[f];
  int st = 0;
  char* d = abi::__cxa_demangle(n.c_str(), nullptr, nullptr, &st);
  std::string s = st == 0 && d ? d : n;
  free(d);
  return s;
}
static std::string where() { return " device=" + std::to_string(g_device); }

extern "C" {
// ---- control
void fake_reset() {
  g_log.clear();
  g_fail = g_allocs = 0;
  g_peak = g_live;
  g_device = 0;
  g_last = cudaSuccess;
}
void fake_set_device(int d) { g_device = d; }
void fake_fail_alloc(long n) { g_fail = n; g_allocs = 0; }   // the n-th from now (0: none)
long fake_allocs() { return g_allocs; }
long long fake_live() { return (long long)g_live; }
long long fake_peak() { return (long long)g_peak; }
long fake_log_size() { return (long)g_log.size(); }
const char* fake_log(long i) { return g_log[i].c_str(); }

// ---- registration
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char* host, char*, const char* name, int, size_t, int, int) {
  names()[host] = name;
}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*,
                            dim3*, dim3*, int*) {
  names()[host] = name;
}

// ---- launches
static std::vector<std::pair<std::pair<dim3, dim3>, std::pair<size_t, cudaStream_t>>> g_conf;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t st) {
  g_conf.push_back({{g, b}, {s, st}});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = g_conf.back().first.first;
  *b = g_conf.back().first.second;
  *s = g_conf.back().second.first;
  *(cudaStream_t*)st = g_conf.back().second.second;
  g_conf.pop_back();
  return cudaSuccess;
}
// positions of the null pointers among the arguments, by the types in the
// demangled name
static std::string null_args(const std::string& sig, void** args) {
  const size_t open = sig.rfind('(') == std::string::npos ? 0 : [&] {
    int depth = 0;
    for (size_t i = sig.size(); i-- > 0;) {   // the parenthesis that matches the last one
      if (sig[i] == ')') ++depth;
      if (sig[i] == '(' && --depth == 0) return i;
    }
    return (size_t)0;
  }();
  std::string out;
  int depth = 0, arg = 0;
  char prev = 0;
  for (size_t i = open + 1; i < sig.size(); ++i) {
    const char c = sig[i];
    if (c == '<' || c == '(') ++depth;
    if ((c == ',' && depth == 0) || (c == ')' && depth == 0)) {
      if (prev == '*' && *(void**)args[arg] == nullptr) out += std::to_string(arg) + ";";
      ++arg;
      if (c == ')') break;
    }
    if (c == '>' || c == ')') --depth;
    if (c != ' ') prev = c;
  }
  return out;
}
static cudaError_t launch(const void* f, dim3 g, dim3 b, void** args) {
  if (g.x == 0 || g.y == 0 || g.z == 0 || g.x > 0x7fffffffu || g.y > 65535u || g.z > 65535u ||
      b.x * b.y * b.z == 0 || b.x * b.y * b.z > 1024) {
    g_last = cudaErrorInvalidConfiguration;
    return g_last;
  }
  const std::string s = demangled(f);
  g_log.push_back("launch " + s + " null=" + null_args(s, args));
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** a, size_t, cudaStream_t) {
  return launch((const void*)k, g, b, a);
}
cudaError_t cudaLaunchKernel(const void* f, dim3 g, dim3 b, void** a, size_t, cudaStream_t) {
  return launch(f, g, b, a);
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3 g, dim3 b, void** a, size_t, cudaStream_t) {
  return launch(f, g, b, a);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** a) {
  return launch(f, c->gridDim, c->blockDim, a);
}

// ---- memory
cudaError_t cudaMalloc(void** p, size_t n) {
  if (++g_allocs == g_fail) {
    g_last = cudaErrorMemoryAllocation;
    return g_last;
  }
  *p = calloc(1, n ? n : 1);
  if (!*p) return cudaErrorMemoryAllocation;
  g_mem[*p] = n;
  g_live += n;
  if (g_live > g_peak) g_peak = g_live;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  g_live -= g_mem[p];
  g_mem.erase(p);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { *p = calloc(1, n ? n : 1); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
static cudaError_t copy(void* d, const void* s, size_t n) {
  if (n <= (1u << 20)) memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  g_log.push_back("copy on the default stream");
  return copy(d, s, n);
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  if (k == cudaMemcpyDeviceToHost) g_log.push_back("download " + std::to_string(n));
  return copy(d, s, n);
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h,
                              cudaMemcpyKind, cudaStream_t) {
  for (size_t i = 0; i < h; ++i) copy((char*)d + i * dp, (const char*)s + i * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  if (n <= (1u << 20)) memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemset2DAsync(void*, size_t, int, size_t, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpyToSymbol(const void* sym, const void*, size_t, size_t, cudaMemcpyKind) {
  g_log.push_back("symbol " + names()[sym] + where());
  return cudaSuccess;
}
cudaError_t cudaMemcpyToSymbolAsync(const void* sym, const void*, size_t, size_t, cudaMemcpyKind,
                                    cudaStream_t) {
  g_log.push_back("symbol " + names()[sym] + " async" + where());
  return cudaSuccess;
}
cudaError_t cudaMemcpyFromSymbolAsync(void* d, const void*, size_t n, size_t, cudaMemcpyKind,
                                      cudaStream_t) {
  memset(d, 0, n);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* sym) { *p = (void*)sym; return cudaSuccess; }

// ---- device and function attributes
cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152
       : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  memset(a, 0, sizeof(*a));
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int) {
  g_log.push_back("attribute " + std::to_string((int)a) + " " + demangled(f) + where());
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = 1;
  return cudaSuccess;
}

// ---- streams, events, errors
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = (cudaStream_t)malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  g_log.push_back(s ? "sync own" : "sync default");
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { *t = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
}
