// A CUDA runtime without a GPU, for tests of the library's host code on the CPU: preloaded
// before libforte_gpu.so, it takes the place of the runtime calls the library makes.
// Device memory is host memory, kernels are not run: a launch is recorded with the
// kernel's name and the positions of its null pointer arguments.  The n-th allocation or
// asynchronous copy from now on can be made to fail (fake_fail_at, fake_fail_copy_at), and
// live allocations are counted.
#include <cuda_runtime_api.h>
#include <cxxabi.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
struct Kernel {
  std::string name;        // demangled, without arguments
  std::vector<bool> ptr;   // which parameters are pointers
};
struct State {
  std::map<const void *, Kernel> kernels;
  std::map<void *, size_t> live;
  long long allocs = 0, fail_at = -1, copies = 0, fail_copy_at = -1;
  cudaError_t last = cudaSuccess;
  std::string log;
  dim3 grid, block;
  size_t smem = 0;
  cudaStream_t stream = nullptr;
};
State &st() {
  static State *s = new State;  // outlives the library's static destructors
  return *s;
}

Kernel parse(const char *mangled) {
  Kernel k;
  int rc = 0;
  char *d = abi::__cxa_demangle(mangled, nullptr, nullptr, &rc);
  std::string s = rc == 0 ? d : mangled;
  free(d);
  // "[void ]name<...>(a, b, ...)": the last top-level parenthesis opens the parameters
  int depth = 0;
  size_t open = s.size(), end = s.rfind(')');
  for (size_t i = 0; i < s.size(); ++i) {
    if (s[i] == '<') ++depth;
    if (s[i] == '>') --depth;
    if (s[i] == '(' && depth == 0 && s.compare(i, 21, "(anonymous namespace)") != 0) {
      open = i;
      break;
    }
  }
  k.name = s.substr(0, open);
  if (k.name.compare(0, 5, "void ") == 0) k.name = k.name.substr(5);
  if (open >= s.size()) return k;
  std::string arg;
  depth = 0;
  for (size_t i = open + 1; i <= end; ++i) {
    if ((s[i] == ',' && depth == 0) || i == end) {
      if (!arg.empty()) k.ptr.push_back(arg.find('*') != std::string::npos);
      arg.clear();
      continue;
    }
    if (s[i] == '<') ++depth;
    if (s[i] == '>') --depth;
    arg += s[i];
  }
  return k;
}

cudaError_t launch(const void *fun, void **args) {
  auto it = st().kernels.find(fun);
  std::string line = it == st().kernels.end() ? "?" : it->second.name;
  if (it != st().kernels.end())
    for (size_t i = 0; i < it->second.ptr.size(); ++i)
      if (it->second.ptr[i] && *(void **)args[i] == nullptr) line += " null" + std::to_string(i);
  st().log += line + "\n";
  return cudaSuccess;
}
cudaError_t fail(cudaError_t e) { return st().last = e; }
cudaError_t allocate(void **p, size_t n) {
  State &s = st();
  if (++s.allocs == s.fail_at) {
    s.fail_at = -1;
    return fail(cudaErrorMemoryAllocation);
  }
  *p = calloc(n ? n : 1, 1);
  s.live[*p] = n;
  return cudaSuccess;
}
cudaError_t release(void *p) {
  if (!p) return cudaSuccess;
  if (!st().live.erase(p)) return fail(cudaErrorInvalidValue);
  free(p);
  return cudaSuccess;
}
int no_tensor_map(...) { return 0; }  // cuTensorMapEncodeTiled
}  // namespace

extern "C" {
// ---- for the tests
void fake_fail_at(long long n) { st().fail_at = n < 0 ? -1 : st().allocs + n; }
void fake_fail_copy_at(long long n) { st().fail_copy_at = n < 0 ? -1 : st().copies + n; }
long long fake_allocs() { return st().allocs; }
long long fake_live() { return (long long)st().live.size(); }
int fake_last_error() { return (int)st().last; }
const char *fake_log() { return st().log.c_str(); }
void fake_clear_log() { st().log.clear(); }

// ---- launches
void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *fun, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
  st().kernels[fun] = parse(name);
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  st().grid = g;
  st().block = b;
  st().smem = smem;
  st().stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *s) {
  *g = st().grid;
  *b = st().block;
  *smem = st().smem;
  *(cudaStream_t *)s = st().stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fun) {
  *k = (cudaKernel_t)fun;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **args, size_t, cudaStream_t) {
  return launch((const void *)k, args);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *fun, void **args) { return launch(fun, args); }

// ---- memory
cudaError_t cudaMalloc(void **p, size_t n) { return allocate(p, n); }
cudaError_t cudaFree(void *p) { return release(p); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return allocate(p, n); }
cudaError_t cudaFreeHost(void *p) { return release(p); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
  if (++st().copies == st().fail_copy_at) return fail(cudaErrorInvalidValue);
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) {
  memset(p, v, n);
  return cudaSuccess;
}

// ---- the rest succeeds
cudaError_t cudaGetLastError() {
  const cudaError_t e = st().last;
  st().last = cudaSuccess;
  return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 152;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
  memset(a, 0, sizeof(*a));
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
  *e = (cudaEvent_t)8;
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
  *p = (void *)no_tensor_map;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}
