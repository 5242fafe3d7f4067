// A host-only run of libhp.so on a fake CUDA runtime (this executable's own definitions of the
// runtime's entry points come before the real library's): device memory is host memory, kernels
// do nothing, and one chosen launch is refused as the runtime refuses one, by a returned error
// that stays pending for cudaGetLastError.
//
//   launch_errors DIM N COLUMNS FIRST_KERNEL_ATTRIBUTE
//
// prints for the prior solve of that problem "launches L", then for every one of its L launches
// the solve's status with that launch refused and with none refused afterwards, and the
// launches of the latter.  FIRST_KERNEL_ATTRIBUTE 1: cudaFuncSetAttribute is refused instead.
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include <cuda_runtime_api.h>

#include "hp.h"

static cudaError_t g_last = cudaSuccess;
static long g_launches = 0, g_refuse = -1, g_attr_refuse = 0, g_attr_refused = 0;

static cudaError_t launched() {
  if (g_launches++ != g_refuse) return cudaSuccess;
  return g_last = cudaErrorLaunchOutOfResources;
}
template <class T> static T handle() {  // a distinct non-null handle
  static uintptr_t next = 16;
  return reinterpret_cast<T>(next += 16);
}

extern "C" {
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaPeekAtLastError() { return g_last; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorLaunchOutOfResources ? "refused" : "other"; }

// kernels
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) { return launched(); }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) { return launched(); }
static dim3 c_grid, c_block;
static size_t c_shm;
static cudaStream_t c_stream;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t shm, cudaStream_t st) {
  c_grid = g;
  c_block = b;
  c_shm = shm;
  c_stream = st;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *shm, cudaStream_t *st) {
  *g = c_grid;
  *b = c_block;
  *shm = c_shm;
  *st = c_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *) {
  *k = handle<cudaKernel_t>();
  return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *) {
  static void *h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) {
  if (!g_attr_refuse) return cudaSuccess;
  ++g_attr_refused;
  return g_last = cudaErrorInvalidValue;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}

// memory
cudaError_t cudaMalloc(void **p, size_t n) {
  *p = calloc(n ? n : 1, 1);
  return *p ? cudaSuccess : g_last = cudaErrorMemoryAllocation;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void *p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t) {
  for (size_t i = 0; i < h; ++i) memcpy((char *)d + i * dp, (const char *)s + i * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaMemcpyFromSymbol(void *d, const void *, size_t n, size_t, cudaMemcpyKind) { return cudaMemset(d, 0, n); }
cudaError_t cudaMemcpyFromSymbolAsync(void *d, const void *, size_t n, size_t, cudaMemcpyKind, cudaStream_t) {
  return cudaMemset(d, 0, n);
}
cudaError_t cudaMemcpyToSymbol(const void *, const void *, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyToSymbolAsync(const void *, const void *, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
  return cudaSuccess;
}

// device, streams, events
cudaError_t cudaGetDevice(int *d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) {
  *s = handle<cudaStream_t>();
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) {
  *e = handle<cudaEvent_t>();
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}

// capture and graphs: accepted, nothing runs
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *,
                                          size_t, cudaStreamCaptureMode) {
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaSuccess; }
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, cudaStreamCaptureStatus *st, unsigned long long *, cudaGraph_t *,
                                     const cudaGraphNode_t **deps, const cudaGraphEdgeData **, size_t *n) {
  static cudaGraphNode_t leaf = handle<cudaGraphNode_t>();
  *st = cudaStreamCaptureStatusActive;
  *deps = &leaf;
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaGraphCreate(cudaGraph_t *g, unsigned) {
  *g = handle<cudaGraph_t>();
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle *h, cudaGraph_t, unsigned, unsigned) {
  *h = 1;
  return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t *n, cudaGraph_t, const cudaGraphNode_t *, const cudaGraphEdgeData *,
                             size_t, cudaGraphNodeParams *p) {
  static cudaGraph_t body = handle<cudaGraph_t>();
  *n = handle<cudaGraphNode_t>();
  p->conditional.phGraph_out = &body;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t, unsigned long long) {
  *x = handle<cudaGraphExec_t>();
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
}

int main(int argc, char **argv) {
  if (argc != 5) return 2;
  hp_problem_desc d{};
  d.dim = atoi(argv[1]);
  d.N = atoi(argv[2]);
  d.gamma = 0.1;
  d.delta = 0.5;
  d.sigma = 0.01;
  d.precision = HP_FP32_IR;
  d.rtol = 1e-10;
  d.max_iter = 100;
  const int cols = atoi(argv[3]), attribute = atoi(argv[4]);
  long n = 1;
  for (int a = 0; a < d.dim; ++a) n *= d.N + 1;
  std::vector<double> B(n * cols), X(n * cols);
  long launches = -1;
  for (long k = -1; k < (attribute ? 0 : launches < 0 ? 1 : launches); ++k) {
    hp_problem *P = nullptr;
    g_refuse = -1;
    g_attr_refuse = 0;
    if (hp_problem_create(&d, &P)) {
      printf("create: %s\n", hp_last_error());
      return 1;
    }
    auto solve = [&]() { return hp_prior_solve(P, B.data(), n, X.data(), n, cols, nullptr); };
    g_launches = 0;
    if (attribute && k < 0) g_attr_refuse = 1;
    g_refuse = attribute ? -1 : k;
    const int first = solve();
    const long l1 = g_launches;
    g_launches = 0;
    g_refuse = -1;
    g_attr_refuse = 0;
    const int second = solve();
    if (attribute) {
      printf("attribute %ld %d %d\n", g_attr_refused, first, second);
    } else if (k < 0) {
      launches = l1;
      printf("launches %ld\n", launches);
    } else {
      printf("%ld %d %d %ld\n", k, first, second, g_launches);
    }
    hp_problem_destroy(P);
  }
  return 0;
}
