/* A CUDA runtime without a device, for tests of the library's host code: device memory is host memory, kernels do nothing, and what is
 * called, copied, launched or captured is written down as a line of text.  fake_fail makes the n-th next call of one function fail. */
#include <cuda_runtime_api.h>
#include <stdarg.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

static char log_text[1 << 20];
static size_t log_len;
static int capturing, captured, fail_in;
static char fail_name[64];
static cudaError_t last_error;
static struct { const void* host; const char* name; size_t max_smem; } kernels[512];
static int n_kernels;
static struct { uintptr_t lo, hi; } pinned[64];
static int n_pinned;

static void note(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  if (log_len + 512 < sizeof(log_text)) log_len += (size_t)vsnprintf(log_text + log_len, 512, fmt, ap);
  va_end(ap);
}
static cudaError_t done(const char* name) {
  if (fail_in > 0 && !strcmp(name, fail_name) && --fail_in == 0) {
    note("failed %s\n", name);
    return cudaErrorInvalidValue;
  }
  return cudaSuccess;
}
const char* fake_log(void) { return log_text; }
void fake_reset(void) { log_len = 0; log_text[0] = 0; fail_in = 0; }
void fake_fail(const char* name, int nth) { snprintf(fail_name, sizeof(fail_name), "%s", name); fail_in = nth; }
/* a range of page-locked memory of the caller's; the 64 newest are known */
void fake_pinned(void* p, size_t n) {
  pinned[n_pinned % 64].lo = (uintptr_t)p;
  pinned[n_pinned++ % 64].hi = (uintptr_t)p + n;
}

void fake_unpin(void) { n_pinned = 0; }

void** __cudaRegisterFatBinary(void* f) { (void)f; static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void** h, char* v, char* a, const char* n, int e, size_t s, int c, int g) { (void)h; (void)v; (void)a; (void)n; (void)e; (void)s; (void)c; (void)g; }
void __cudaRegisterFunction(void** h, const char* host, char* dev, const char* name, int lim, uint3* t, uint3* b, dim3* bd, dim3* gd, int* w) {
  (void)h; (void)dev; (void)lim; (void)t; (void)b; (void)bd; (void)gd; (void)w;
  if (n_kernels < 512) {
    kernels[n_kernels].host = host;
    kernels[n_kernels].max_smem = 47 * 1024;   /* 48 KB without asking, static variables (up to 1 KB here) included */
    kernels[n_kernels++].name = name;
  }
}
static struct { dim3 grid, block; size_t smem; void* stream; } pushed;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* s) {
  pushed.grid = grid; pushed.block = block; pushed.smem = smem; pushed.stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
  *grid = pushed.grid; *block = pushed.block; *smem = pushed.smem; *(void**)s = pushed.stream;
  return cudaSuccess;
}
static cudaError_t launch(const char* call, const void* func, dim3 grid, size_t smem) {
  cudaError_t e = done(call);
  const char* name = "?";
  for (int i = 0; i < n_kernels; ++i)
    if (kernels[i].host == func) {
      name = kernels[i].name;
      if (smem > kernels[i].max_smem) e = cudaErrorInvalidValue;
    }
  if (e != cudaSuccess) last_error = e;
  if (e == cudaSuccess) {
    captured += capturing;
    note("%s %s grid %u %u %u smem %zu\n", capturing ? "capture" : "launch", name, grid.x, grid.y, grid.z, smem);
  }
  return e;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* func, void** args) { (void)args; return launch("cudaLaunchKernel", func, c->gridDim, c->dynamicSmemBytes); }
cudaError_t cudaLaunchKernel(const void* func, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t s) {
  (void)block; (void)args; (void)s;
  return launch("cudaLaunchKernel", func, grid, smem);
}

cudaError_t cudaMalloc(void** p, size_t n) { *p = aligned_alloc(256, (n + 255) / 256 * 256); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) { (void)k; memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
  cudaError_t e = done("cudaMemcpyAsync");
  (void)st;
  if (e != cudaSuccess) return e;
  memcpy(d, s, n);
  note("copy %s %zu from %p to %p\n", k == cudaMemcpyHostToDevice ? "in" : "out", n, s, d);
  return e;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t s) { (void)s; memset(d, v, n); note("clear %p %zu\n", d, n); return cudaSuccess; }
static cudaError_t handle(void* out) { *(void**)out = malloc(8); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return handle(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned f) { (void)f; return handle(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { (void)a; (void)b; *ms = 0.125f; return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)s; note("record %p\n", (void*)e); return done("cudaEventRecord"); }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { (void)f; return handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; note("drain\n"); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)s; (void)f; note("wait %p\n", (void*)e); return done("cudaStreamWaitEvent"); }
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s; (void)m; capturing = 1; captured = 0; return done("cudaStreamBeginCapture"); }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) { (void)s; capturing = 0; handle(g); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long f) { (void)g; (void)f; handle(x); *(int*)*x = captured; return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) {
  cudaError_t e = done("cudaGraphLaunch");
  (void)s;
  if (e == cudaSuccess) note("replay %d\n", *(int*)x);
  return e;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { free(g); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { free(x); return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) {
  for (int i = 0; i < n_kernels; ++i)
    if (kernels[i].host == f && a == cudaFuncAttributeMaxDynamicSharedMemorySize) kernels[i].max_smem = (size_t)v;
  return v <= 227 * 1024 ? cudaSuccess : cudaErrorInvalidValue;
}
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { (void)d; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { (void)a; (void)d; *v = 148; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(struct cudaDeviceProp* p, int d) {
  (void)d;
  memset(p, 0, sizeof(*p));
  p->major = 10;
  p->multiProcessorCount = 148;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) { (void)f; (void)c; *n = 74; return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "made by the test"; }
cudaError_t cudaGetLastError(void) {
  const cudaError_t e = last_error;
  last_error = cudaSuccess;
  return e;
}

static int encode_tiled(void) { return 0; }
static int pointer_attribute(void* out, int what, uintptr_t p) {
  (void)what;
  for (int i = 0; i < 64 && i < n_pinned; ++i)
    if (p >= pinned[i].lo && p < pinned[i].hi) { *(uintptr_t*)out = pinned[i].lo; return 0; }
  return 1;
}
static unsigned char symbols[4][1 << 16] __attribute__((aligned(256)));   /* where a context keeps the library's one array */
/* A context is gone and another current: kernels are as they were loaded.  No two have the same number. */
static unsigned long long context_id = 7;
void fake_new_context(void) {
  ++context_id;
  for (int i = 0; i < n_kernels; ++i) kernels[i].max_smem = 47 * 1024;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
  (void)s;
  *p = symbols[context_id % 4];
  note("symbol %p\n", *p);
  return cudaSuccess;
}
static int context_number(void* ctx, unsigned long long* id) { (void)ctx; *id = context_id; return 0; }
cudaError_t cudaGetDriverEntryPoint(const char* name, void** f, unsigned long long flags, enum cudaDriverEntryPointQueryResult* q) {
  (void)flags;
  *f = !strcmp(name, "cuPointerGetAttribute") ? (void*)pointer_attribute : !strcmp(name, "cuCtxGetId") ? (void*)context_number : (void*)encode_tiled;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
