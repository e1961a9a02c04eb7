// A stand-in for the CUDA runtime, preloaded over libcudart: memory is the host's, copies are copies,
// kernels are not run but their launches are checked as the driver checks them and written down.  For
// tests of what the library's host code does with devices, contexts, limits and refused calls.
#define _GNU_SOURCE
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>

#define DEVICES 2
#define MOST 4096
#define OUT __attribute__((visibility("default")))

static __thread int t_dev = 0;
static __thread cudaError_t t_last = cudaSuccess;
static unsigned long long g_ctx[DEVICES] = {1000, 2000};
static struct { const void* fn; const char* name; int limit[DEVICES]; unsigned long long ctx[DEVICES]; } g_fn[MOST];
static int g_fns = 0;
static char g_log[1 << 20];
static size_t g_logged = 0, g_most_bytes = 0;
static char g_refuse[128];
static int g_nodes = 0, g_symbols = 0;
static float g_event_ms = 1.0f;

static cudaError_t err(cudaError_t e) { if (e) t_last = e; return e; }

// ---- the tests' side
OUT void fake_device(int d) { t_dev = d; }
OUT void fake_reset(int d) { g_ctx[d] += 1; }                                    // as by cudaDeviceReset
OUT void fake_refuse(const char* s) { snprintf(g_refuse, sizeof g_refuse, "%s", s); }  // launches of these kernels
OUT void fake_memory(size_t most) { g_most_bytes = most; }                        // of one allocation; 0: any
OUT const char* fake_log(void) { return g_log; }
OUT void fake_clear(void) { g_logged = 0; g_log[0] = 0; }

static int find(const void* fn) {
  for (int i = 0; i < g_fns; ++i)
    if (g_fn[i].fn == fn) return i;
  return -1;
}

// ---- registration and launches
OUT void** __cudaRegisterFatBinary(void* p) { static void* h; (void)p; return &h; }
OUT void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
OUT void __cudaUnregisterFatBinary(void** h) { (void)h; }
OUT void __cudaRegisterVar(void** h, char* v, char* a, const char* n, int e, size_t s, int c, int g) {
  (void)h; (void)v; (void)a; (void)n; (void)e; (void)s; (void)c; (void)g;
}
OUT void __cudaRegisterFunction(void** h, const char* fn, char* dfn, const char* name, int tl, uint3* t, uint3* b, void* bd,
                                void* gd, int* w) {
  (void)h; (void)dfn; (void)tl; (void)t; (void)b; (void)bd; (void)gd; (void)w;
  if (g_fns < MOST) { g_fn[g_fns].fn = fn; g_fn[g_fns].name = name; ++g_fns; }
}
static __thread struct { struct dim3 g, b; size_t s; void* st; } t_call;
OUT unsigned __cudaPushCallConfiguration(struct dim3 g, struct dim3 b, size_t s, void* st) {
  t_call.g = g; t_call.b = b; t_call.s = s; t_call.st = st;
  return 0;
}
OUT cudaError_t __cudaPopCallConfiguration(struct dim3* g, struct dim3* b, size_t* s, void* st) {
  *g = t_call.g; *b = t_call.b; *s = t_call.s; *(void**)st = t_call.st;
  return cudaSuccess;
}
OUT cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) { *k = (cudaKernel_t)fn; return cudaSuccess; }
OUT cudaError_t __cudaLaunchKernel(cudaKernel_t k, struct dim3 g, struct dim3 b, void** a, size_t smem, cudaStream_t s) {
  (void)a; (void)s;
  const int i = find((const void*)k);
  const char* name = i >= 0 ? g_fn[i].name : "?";
  int limit = 48 * 1024;
  if (i >= 0 && g_fn[i].ctx[t_dev] == g_ctx[t_dev] && g_fn[i].limit[t_dev] > limit) limit = g_fn[i].limit[t_dev];
  cudaError_t e = cudaSuccess;
  if (!g.x || !g.y || !g.z || g.x > 0x7fffffffu || g.y > 65535 || g.z > 65535 || !b.x || b.x * b.y * b.z > 1024)
    e = cudaErrorInvalidConfiguration;
  if ((int)smem > limit) e = cudaErrorInvalidValue;
  if (g_refuse[0] && strstr(name, g_refuse)) e = cudaErrorLaunchOutOfResources;
  g_nodes += e == cudaSuccess;
  if (g_logged + 512 < sizeof g_log)
    g_logged += snprintf(g_log + g_logged, 512, "%d %d %.200s %u %u %u %u %zu\n", (int)e, t_dev, name, g.x, g.y, g.z, b.x, smem);
  return err(e);
}
OUT cudaError_t cudaFuncSetAttribute(const void* fn, enum cudaFuncAttribute a, int v) {
  const int i = find(fn);
  if (i < 0 || (a == cudaFuncAttributeMaxDynamicSharedMemorySize && v > 232448)) return err(cudaErrorInvalidValue);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) { g_fn[i].limit[t_dev] = v; g_fn[i].ctx[t_dev] = g_ctx[t_dev]; }
  return cudaSuccess;
}

// ---- devices and the driver's entry points
static int ctx_current(void** c) { *c = &g_ctx[t_dev]; return 0; }  // a reset gives the same address
static int ctx_id(void* c, unsigned long long* id) { *id = *(unsigned long long*)c; return 0; }
static int encode(void) { return 0; }
OUT cudaError_t cudaGetDriverEntryPointByVersion(const char* n, void** p, unsigned v, unsigned long long f,
                                                 enum cudaDriverEntryPointQueryResult* q) {
  (void)v; (void)f;
  *p = !strcmp(n, "cuCtxGetCurrent") ? (void*)ctx_current : !strcmp(n, "cuCtxGetId") ? (void*)ctx_id
     : !strcmp(n, "cuTensorMapEncodeTiled") ? (void*)encode : NULL;
  if (q) *q = *p ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
OUT cudaError_t cudaGetDevice(int* d) { *d = t_dev; return cudaSuccess; }
OUT cudaError_t cudaGetDeviceCount(int* n) { *n = DEVICES; return cudaSuccess; }
OUT cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) {
  (void)d;
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
OUT cudaError_t cudaGetDeviceProperties(struct cudaDeviceProp* p, int d) {
  (void)d;
  memset(p, 0, sizeof *p);
  strcpy(p->name, "fake");
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
OUT cudaError_t cudaGetLastError(void) { cudaError_t e = t_last; t_last = cudaSuccess; return e; }
OUT cudaError_t cudaPeekAtLastError(void) { return t_last; }
OUT int fake_symbols(void) { return g_symbols; }  // addresses asked for
OUT cudaError_t cudaGetSymbolAddress(void** p, const void* s) {
  static void* mem;
  (void)s;
  ++g_symbols;
  if (!mem) mem = mmap(NULL, 128u << 20, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  *p = mem;
  return cudaSuccess;
}

// ---- memory (never returned to the system: the tests are short)
static cudaError_t take(void** p, size_t n) {
  *p = NULL;
  if (g_most_bytes && n > g_most_bytes) return err(cudaErrorMemoryAllocation);
  *p = mmap(NULL, n + 4096, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (*p == MAP_FAILED) { *p = NULL; return err(cudaErrorMemoryAllocation); }
  if (g_logged + 64 < sizeof g_log) g_logged += snprintf(g_log + g_logged, 64, "alloc %zu\n", n);
  return cudaSuccess;
}
OUT cudaError_t cudaMalloc(void** p, size_t n) { return take(p, n); }
OUT cudaError_t cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; return take(p, n); }
OUT cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t s) { (void)s; return take(p, n); }
OUT cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t m, cudaStream_t s) { (void)m; (void)s; return take(p, n); }
OUT cudaError_t cudaFree(void* p) { (void)p; return cudaSuccess; }
OUT cudaError_t cudaFreeHost(void* p) { (void)p; return cudaSuccess; }
OUT cudaError_t cudaFreeAsync(void* p, cudaStream_t s) { (void)p; (void)s; return cudaSuccess; }
OUT cudaError_t cudaMemPoolCreate(cudaMemPool_t* m, const struct cudaMemPoolProps* q) { (void)q; *m = (cudaMemPool_t)&g_ctx; return cudaSuccess; }
OUT cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t m, enum cudaMemPoolAttr a, void* v) { (void)m; (void)a; (void)v; return cudaSuccess; }
OUT cudaError_t cudaMemPoolTrimTo(cudaMemPool_t m, size_t n) { (void)m; (void)n; return cudaSuccess; }
OUT cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) { (void)k; memmove(d, s, n); return cudaSuccess; }
OUT cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t t) { (void)k; (void)t; memmove(d, s, n); return cudaSuccess; }
OUT cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, enum cudaMemcpyKind k, cudaStream_t t) {
  (void)k; (void)t;
  for (size_t i = 0; i < h; ++i) memmove((char*)d + i * dp, (const char*)s + i * sp, w);
  return cudaSuccess;
}
OUT cudaError_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
OUT cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t t) { (void)t; memset(d, v, n); return cudaSuccess; }

// ---- streams, events, graphs
OUT cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { (void)f; *s = (cudaStream_t)&g_nodes; return cudaSuccess; }
OUT cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return cudaSuccess; }
OUT cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; return cudaSuccess; }
OUT cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)s; (void)e; (void)f; return cudaSuccess; }
OUT cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)&g_log; return cudaSuccess; }
OUT cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned f) { (void)f; *e = (cudaEvent_t)&g_log; return cudaSuccess; }
OUT cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
OUT cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e; (void)s; return cudaSuccess; }
OUT cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
OUT cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {  // each reading a little shorter
  (void)a; (void)b;
  *ms = g_event_ms *= 0.999f;
  return cudaSuccess;
}
OUT cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode m) { (void)s; (void)m; g_nodes = 0; return cudaSuccess; }
OUT cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) { (void)s; *g = (cudaGraph_t)&g_fns; return cudaSuccess; }
OUT cudaError_t cudaGraphGetNodes(cudaGraph_t g, cudaGraphNode_t* n, size_t* count) { (void)g; (void)n; *count = g_nodes; return cudaSuccess; }
OUT cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long f) { (void)g; (void)f; *x = (cudaGraphExec_t)&g_fn; return cudaSuccess; }
OUT cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) { (void)x; (void)s; return cudaSuccess; }
OUT cudaError_t cudaGraphDestroy(cudaGraph_t g) { (void)g; return cudaSuccess; }
OUT cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { (void)x; return cudaSuccess; }
