/* A CUDA runtime without a GPU, for tests of the library's host logic: device memory is host memory, copies and
 * memsets are done, kernels are recorded by name and not run, and the n-th call of a chosen kind can be made to
 * fail.  Asynchronous copies to the host deliver doubles of 1 (valid densities) in place of what the kernels would have
 * written.  The library's objects are linked with this file instead of the CUDA runtime. */
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <string.h>

enum { MAX_FUNCS = 4096, MAX_LOG = 1 << 16 };
static const void *g_fun[MAX_FUNCS];
static char g_name[MAX_FUNCS][192];
static char g_dep[MAX_FUNCS][208]; /* the same, launched as a programmatic dependent */
static int g_nfun;

/* Recorded calls: kernel names, and "graph launch". */
static const char *g_log[MAX_LOG];
static int g_nlog;
static char g_fail_what[64];
static int g_fail_in;    /* calls of that kind still served before one fails; < 0: none */
static int g_capturing;  /* what cudaStreamIsCapturing says */
static int g_last;
static dim3 g_grid, g_block;

void fake_reset(void) { g_nlog = 0, g_fail_in = -1, g_capturing = 0, g_last = 0; }
/* Calls named `what` (a runtime function, or "kernel" for any launch): the next `after` are served, then one fails. */
void fake_fail(const char *what, int after) {
  snprintf(g_fail_what, sizeof g_fail_what, "%s", what);
  g_fail_in = after;
}
void fake_capturing(int on) { g_capturing = on; }
int fake_calls(void) { return g_nlog; }
const char *fake_call(int k) { return g_log[k]; }

static cudaError_t result(const char *what) {
  if (g_fail_in >= 0 && !strcmp(what, g_fail_what) && g_fail_in-- == 0) return (cudaError_t)(g_last = cudaErrorUnknown);
  return cudaSuccess;
}
static void record(const char *s) {
  if (g_nlog < MAX_LOG) g_log[g_nlog++] = s;
}
static cudaError_t launch(const void *f, int dep) {
  const cudaError_t e = result("kernel");
  if (e != cudaSuccess) return e;
  for (int k = 0; k < g_nfun; ++k)
    if (g_fun[k] == f) {
      record(dep ? g_dep[k] : g_name[k]);
      return cudaSuccess;
    }
  return (cudaError_t)(g_last = cudaErrorInvalidDeviceFunction);
}

/* what the compiler's host code calls */
void **__cudaRegisterFatBinary(void *f) { return (void **)f; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int limit, uint3 *tid, uint3 *bid,
                            dim3 *bd, dim3 *gd, int *ws) {
  (void)h, (void)dev, (void)limit, (void)tid, (void)bid, (void)bd, (void)gd, (void)ws;
  if (g_nfun == MAX_FUNCS) return;
  g_fun[g_nfun] = host;
  snprintf(g_name[g_nfun], sizeof g_name[0], "%s", name);
  snprintf(g_dep[g_nfun], sizeof g_dep[0], "%s (dependent)", g_name[g_nfun]);
  g_nfun++;
}
void __cudaRegisterVar(void **h, char *host, char *dev, const char *name, int ext, size_t size, int c, int g) {
  (void)h, (void)host, (void)dev, (void)name, (void)ext, (void)size, (void)c, (void)g;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st *st) {
  (void)smem, (void)st;
  g_grid = g, g_block = b;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *smem, void *st) {
  *g = g_grid, *b = g_block, *smem = 0, *(void **)st = 0;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void **args, size_t smem, cudaStream_t st) {
  (void)g, (void)b, (void)args, (void)smem, (void)st;
  return launch((const void *)k, 0);
}

cudaError_t cudaLaunchKernel(const void *f, dim3 g, dim3 b, void **args, size_t smem, cudaStream_t st) {
  return __cudaLaunchKernel((cudaKernel_t)f, g, b, args, smem, st);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
  (void)args;
  return launch(f, c->numAttrs > 0);
}
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr a, int d) {
  (void)d;
  return *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1, cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) { return (void)f, (void)a, (void)v, cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int b, size_t s) {
  (void)f, (void)b, (void)s;
  return *n = 2, cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, size_t s, unsigned fl) {
  (void)fl;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, b, s);
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "injected"; }
cudaError_t cudaGetLastError(void) {
  const int e = g_last;
  g_last = 0;
  return (cudaError_t)e;
}
cudaError_t cudaGetSymbolAddress(void **p, const void *s) { return *p = (void *)s, cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k) { return (void)k, memmove(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
  (void)st;
  const cudaError_t e = result("cudaMemcpyAsync");
  if (e != cudaSuccess || k != cudaMemcpyDeviceToHost) return e == cudaSuccess ? cudaMemcpy(d, s, n, k) : e;
  for (size_t i = 0; i < n / sizeof(double); ++i) ((double *)d)[i] = 1.0;
  return cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) { return memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st) { return (void)st, cudaMemset(d, v, n); }
cudaError_t cudaStreamSynchronize(cudaStream_t st) { return (void)st, cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *st, unsigned f) {
  (void)f;
  *st = (cudaStream_t)1;
  return result("cudaStreamCreateWithFlags");
}
cudaError_t cudaStreamDestroy(cudaStream_t st) { return (void)st, cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t st, enum cudaStreamCaptureStatus *c) {
  (void)st;
  return *c = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t st, enum cudaStreamCaptureMode m) {
  (void)st, (void)m;
  return result("cudaStreamBeginCapture");
}
cudaError_t cudaStreamEndCapture(cudaStream_t st, cudaGraph_t *g) { return (void)st, *g = (cudaGraph_t)1, cudaSuccess; }
cudaError_t cudaGraphCreate(cudaGraph_t *g, unsigned f) { return (void)f, *g = (cudaGraph_t)1, cudaSuccess; }
cudaError_t cudaGraphAddKernelNode(cudaGraphNode_t *n, cudaGraph_t g, const cudaGraphNode_t *d, size_t nd,
                                   const struct cudaKernelNodeParams *p) {
  (void)g, (void)d, (void)nd;
  *n = (cudaGraphNode_t)1;
  return launch(p->func, 0);
}
cudaError_t cudaGraphAddMemsetNode(cudaGraphNode_t *n, cudaGraph_t g, const cudaGraphNode_t *d, size_t nd,
                                   const struct cudaMemsetParams *p) {
  (void)g, (void)d, (void)nd, (void)p;
  return *n = (cudaGraphNode_t)1, cudaSuccess;
}
cudaError_t cudaGraphKernelNodeSetAttribute(cudaGraphNode_t n, cudaLaunchAttributeID a, const cudaLaunchAttributeValue *v) {
  return (void)n, (void)a, (void)v, cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t g, unsigned long long f) {
  (void)g, (void)f;
  *e = 0;
  const cudaError_t r = result("cudaGraphInstantiate");
  if (r == cudaSuccess) *e = (cudaGraphExec_t)1;
  return r;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t st) {
  (void)st;
  if (!e) return cudaErrorInvalidValue;
  const cudaError_t r = result("cudaGraphLaunch");
  if (r == cudaSuccess) record("graph launch");
  return r;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return (void)g, cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { return (void)e, cudaSuccess; }
