/* A stand-in for the CUDA runtime, linked with the library's objects to run its host code without a GPU.
 * Device memory is host memory, kernels do nothing, and every call succeeds but the one that
 * fake_fail_at names.  It records what the tests ask about: work left on a stream that nothing orders
 * before a free, and attribute calls made inside a stream capture. */
#include <stddef.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

enum { NS = 64, OK = 0, FAILED = 1 };
typedef struct { unsigned x, y, z; } dim3;
typedef struct { long dep[NS]; } event;
typedef void (*hook_fn)(const char* kernel, void** args);

/* stream t's launches are numbered seq[t]; dep[s][t]: those that come before whatever stream s does next,
 * host[t]: those the host has waited for; shared[t]: t takes part in an event wait */
static long seq[NS], dep[NS][NS], host[NS];
static int shared[NS], nstreams, capturing, last_error, attr_in_capture, graphs, unordered_frees;
static long countdown = -1;
static hook_fn hook;
static struct { const void* fn; char name[256]; } kernels[8192];
static int nkernels;

int fake_unordered_frees(void) { return unordered_frees; }
int fake_attr_in_capture(void) { return attr_in_capture; }
int fake_graphs(void) { return graphs; }
void fake_hook(hook_fn h) { hook = h; }
/* the n-th call from here on (n >= 1) that allocates, launches, forks or joins fails; 0: none */
void fake_fail_at(long n) {
  countdown = n > 0 ? n : -1;
}
static int fails(void) {
  if (countdown <= 0 || --countdown > 0) return OK;
  countdown = -1;
  return last_error = FAILED;
}
static int id(const void* s) { return (int)(uintptr_t)s % NS; }
static long later(long a, long b) { return a > b ? a : b; }

/* ---- registration and launches */
void** __cudaRegisterFatBinary(void* f) { static void* h; (void)f; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void** h, char* v, char* d, const char* n, int e, size_t s, int c, int g) {
  (void)h, (void)v, (void)d, (void)n, (void)e, (void)s, (void)c, (void)g;
}
void __cudaRegisterFunction(void** h, const char* fn, char* d, const char* name, int t, void* a, void* b,
                            void* c, void* e, int* w) {
  (void)h, (void)d, (void)t, (void)a, (void)b, (void)c, (void)e, (void)w;
  if (nkernels == 8192) return;
  kernels[nkernels].fn = fn;
  strncpy(kernels[nkernels++].name, name, 255);
}
static struct { dim3 g, b; size_t sm; void* s; } config;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, void* s) {
  config.g = g, config.b = b, config.sm = sm, config.s = s;
  return 0;
}
int __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* s) {
  *g = config.g, *b = config.b, *sm = config.sm, *(void**)s = config.s;
  return OK;
}
int __cudaGetKernel(const void** k, const void* fn) { *k = fn; return OK; }
int __cudaLaunchKernel(const void* k, dim3 g, dim3 b, void** args, size_t sm, void* s) {
  (void)g, (void)b, (void)sm;
  if (fails()) return FAILED;
  if (capturing) return OK;
  const int t = id(s);
  dep[t][t] = ++seq[t];
  if (hook)
    for (int i = 0; i < nkernels; ++i)
      if (kernels[i].fn == k) hook(kernels[i].name, args);
  return OK;
}
int cudaFuncSetAttribute(const void* f, int a, int v) {
  (void)f, (void)a, (void)v;
  attr_in_capture += capturing;
  return OK;
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int b, size_t s, unsigned l) {
  (void)f, (void)b, (void)s, (void)l;
  *n = 4;
  return OK;
}

/* ---- device, errors, memory */
int cudaGetDevice(int* d) { *d = 0; return OK; }
int cudaSetDevice(int d) { (void)d; return OK; }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)a, (void)d; *v = 152; return OK; }
int cudaDeviceSynchronize(void) { memcpy(host, seq, sizeof(host)); return OK; }
int cudaGetLastError(void) { const int e = last_error; last_error = OK; return e; }
const char* cudaGetErrorString(int e) { return e ? "injected failure" : "no error"; }
int cudaMalloc(void** p, size_t n) {
  if (fails()) return FAILED;
  *p = calloc(1, n);
  return OK;
}
int cudaFree(void* p) { (void)p; return OK; }
int cudaMallocAsync(void** p, size_t n, void* s) { (void)s; return cudaMalloc(p, n); }
int cudaMallocFromPoolAsync(void** p, size_t n, void* pool, void* s) { (void)pool, (void)s; return cudaMalloc(p, n); }
int cudaFreeAsync(void* p, void* s) {
  const int f = id(s);
  (void)p; /* kept: a kernel on an unordered stream would still read it */
  for (int t = 0; t < NS; ++t)
    if (shared[t] && later(host[t], dep[f][t]) < seq[t]) {
      ++unordered_frees;
      break;
    }
  return OK;
}
int cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; return cudaMalloc(p, n); }
int cudaFreeHost(void* p) { (void)p; return OK; }
int cudaMemPoolCreate(void** p, const void* props) { (void)props; *p = &nstreams; return OK; }
int cudaMemPoolSetAttribute(void* p, int a, void* v) { (void)p, (void)a, (void)v; return OK; }
int cudaMemPoolTrimTo(void* p, size_t n) { (void)p, (void)n; return OK; }
int cudaMemcpy(void* d, const void* s, size_t n, int k) { (void)k; memmove(d, s, n); return OK; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int k, void* st) { (void)st; return capturing ? OK : cudaMemcpy(d, s, n, k); }
int cudaMemsetAsync(void* d, int v, size_t n, void* st) { (void)st; if (!capturing) memset(d, v, n); return OK; }
int cudaMemcpyToSymbol(const void* y, const void* s, size_t n, size_t o, int k) { (void)y, (void)s, (void)n, (void)o, (void)k; return OK; }
int cudaGetSymbolAddress(void** p, const void* y) { static char b[1 << 20]; (void)y; *p = b; return OK; }

/* ---- streams, events, graphs */
int cudaStreamCreateWithFlags(void** s, unsigned f) {
  (void)f;
  if (fails()) return FAILED;
  const int t = 1 + nstreams++ % (NS - 1); /* numbers return after NS - 1 streams */
  shared[t] = 0;
  host[t] = seq[t];
  *s = (void*)(uintptr_t)t;
  return OK;
}
int cudaStreamDestroy(void* s) { (void)s; return OK; }
int cudaStreamSynchronize(void* s) {
  for (int t = 0; t < NS; ++t) host[t] = later(host[t], dep[id(s)][t]);
  return OK;
}
int cudaEventCreateWithFlags(void** e, unsigned f) { (void)f; *e = calloc(1, sizeof(event)); return fails(); }
int cudaEventDestroy(void* e) { (void)e; return OK; }
int cudaEventRecord(void* e, void* s) {
  if (fails()) return FAILED;
  memcpy(((event*)e)->dep, dep[id(s)], sizeof(dep[0]));
  return OK;
}
int cudaStreamWaitEvent(void* s, void* e, unsigned f) {
  (void)f;
  if (fails()) return FAILED;
  shared[id(s)] = 1;
  for (int t = 0; t < NS; ++t) dep[id(s)][t] = later(dep[id(s)][t], ((event*)e)->dep[t]);
  return OK;
}
int cudaStreamBeginCapture(void* s, int m) { (void)s, (void)m; capturing = 1; return OK; }
int cudaStreamEndCapture(void* s, void** g) { (void)s; capturing = 0; *g = &graphs; return OK; }
int cudaGraphInstantiate(void** x, void* g, unsigned long long f) { (void)g, (void)f; *x = &graphs; ++graphs; return OK; }
int cudaGraphDestroy(void* g) { (void)g; return OK; }
int cudaGraphExecDestroy(void* x) { (void)x; return OK; }
int cudaGraphLaunch(void* x, void* s) { (void)x, (void)s; return last_error = FAILED; } /* no replay: solves end here */
