// A stand-in for the CUDA runtime on hosts without a GPU: device memory is host memory, kernels are only recorded by
// name, and the few whose results the host code reads back write plausible ones.  Linked with the library's objects it
// lets host tests follow error paths (a refused geometry, an allocation that fails) and see which kernels a call would
// have launched.
#include <cuda_runtime_api.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>

namespace {
std::map<const void *, std::string> &names() {
  static std::map<const void *, std::string> m;
  return m;
}
std::string g_log;
size_t g_live = 0, g_limit = ~(size_t)0;
std::map<void *, size_t> g_blocks;
int g_refuse = 0, g_err_plans = 0;
long long g_tot[4] = {1000, 100, 50, 16};
struct Cfg {
  dim3 g, b;
  size_t s;
  cudaStream_t st;
} g_cfg;

void launched(const void *f, void **args) {
  const std::string &n = names()[f];
  g_log += n + "\n";
  auto is = [&](const char *k) { return n.find(k) != std::string::npos; };
  if (is("k_brick_scan")) {  // slots, entries, pair table, widest brick's orbitals and atoms, work, entries
    long long *out = *(long long **)args[7];
    const long long v[7] = {4, 4, 4, 13, 2, 0, 2};
    memcpy(out, v, sizeof(v));
  } else if (is("k_brick_pairs") && g_refuse) {
    **(unsigned **)args[9] |= 2u;  // GINT_ERRBIT_SKIN
  } else if (is("k_lay_scan")) {   // totals: scratch elements, plan records, list entries
    struct S {
      const long long *in[3];
      long long n[3];
      long long *out[3];
      long long *total;
    };
    long long *t = ((S *)args[0])->total;
    memcpy(t, g_tot, sizeof(g_tot));  // (t[3]: k_lay_count's widest brick)
  } else if (is("k_build_plans") && g_err_plans) {
    **(unsigned **)args[6] |= 4u;
  }
}
}  // namespace

extern "C" {
// controls of the tests
const char *fake_log() { return g_log.c_str(); }
void fake_clear() { g_log.clear(); }
void fake_refuse(int on) { g_refuse = on; }       // the next geometries overlap a pair outside the block set
void fake_plan_error(int on) { g_err_plans = on; }
void fake_limit(size_t bytes) { g_limit = bytes; }  // device memory
size_t fake_live() { return g_live; }
void fake_list_entries(long long n) { g_tot[2] = n; }
void fake_tiles(long long n) { g_tot[0] = n; }  // float32 elements

// what nvcc's host code calls
void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *,
                            int *) {
  names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, cudaStream_t st) {
  g_cfg = Cfg{g, b, s, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *st) {
  *g = g_cfg.g, *b = g_cfg.b, *s = g_cfg.s, *(cudaStream_t *)st = g_cfg.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **args, size_t, cudaStream_t) {
  launched((const void *)k, args);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *f, void **args) {
  launched(f, args);
  return cudaSuccess;
}

cudaError_t cudaMalloc(void **p, size_t n) {
  if (g_live + n > g_limit) return cudaErrorMemoryAllocation;
  *p = calloc(n ? n : 1, 1);
  g_blocks[*p] = n;
  g_live += n;
  return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
  auto it = g_blocks.find(p);
  if (it == g_blocks.end()) return p ? cudaErrorInvalidValue : cudaSuccess;
  g_live -= it->second;
  g_blocks.erase(it);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyToSymbol(const void *, const void *, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *) {
  static double scratch[4096];
  *p = scratch;
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
  *p = calloc(n, 1);
  return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) {
  *d = h;
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 227 * 1024;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
  memset(a, 0, sizeof(*a));
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = nullptr;
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
  *e = nullptr;
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
}
