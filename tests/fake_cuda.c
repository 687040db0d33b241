/* Host stand-in for the CUDA runtime, cuBLAS and cuSOLVER entry points that libfe imports,
 * preloaded by test_host_calls.py: no kernel runs and no GPU is needed.  Every call is written
 * to a log; allocations are host memory of one byte value, copies to and from the host are made, and a
 * launch outside CUDA's documented grid and block limits is refused as the runtime refuses it. */
#define _GNU_SOURCE
#include <stdarg.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>

typedef struct { unsigned x, y, z; } dim3;
enum { OK = 0, E_VALUE = 1, E_NOMEM = 2, E_CONFIG = 9, E_UNSUPPORTED = 801 };

static char* log_buf;
static size_t log_len, log_cap;
static int last_error;
static size_t fail_bytes;        /* allocations of this size fail */
static int fill;                 /* byte that new allocations hold */
static void* capturing;          /* the stream under capture */

static void note(const char* fmt, ...) {
  if (log_len + 512 > log_cap) log_buf = realloc(log_buf, log_cap = 2 * log_cap + 4096);
  va_list a;
  va_start(a, fmt);
  log_len += vsnprintf(log_buf + log_len, 500, fmt, a);
  va_end(a);
  log_buf[log_len++] = '\n';
  log_buf[log_len] = 0;
}
static int fail(int e) { return last_error = e; }

const char* fake_log(void) { return log_buf ? log_buf : ""; }
void fake_reset(void) { log_len = 0; if (log_buf) log_buf[0] = 0; }
void fake_fail_malloc(size_t bytes) { fail_bytes = bytes; }
void fake_fill(int byte) { fill = byte; }

/* ---- memory ---- */
static struct { void* p; size_t n; } blocks[4096];
static int nblocks;
int cudaMalloc(void** p, size_t n) {
  *p = NULL;
  if (fail_bytes && n == fail_bytes) { note("nomem %zu", n); return fail(E_NOMEM); }
  void* q = mmap(NULL, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (q == MAP_FAILED || nblocks == 4096) return fail(E_NOMEM);
  if (fill) memset(q, fill, n);
  blocks[nblocks].p = q;
  blocks[nblocks++].n = n ? n : 1;
  note("malloc %p %zu", q, n);
  *p = q;
  return OK;
}
int cudaFree(void* p) {
  if (!p) return OK;
  note("free %p", p);
  for (int i = 0; i < nblocks; ++i)
    if (blocks[i].p == p) {
      munmap(p, blocks[i].n);
      blocks[i] = blocks[--nblocks];
      return OK;
    }
  return fail(E_VALUE);
}
/* addresses below 1 << 20 belong to no memory, those below 1 << 24 to device 1, others to device 0 */
typedef struct { int type, device; void *dev, *host; long reserved[8]; } PointerAttributes;
int cudaPointerGetAttributes(PointerAttributes* a, const void* p) {
  memset(a, 0, sizeof *a);
  if ((uintptr_t)p < 1u << 20) return OK;
  a->type = 2;
  a->device = (uintptr_t)p < 1u << 24;
  a->dev = (void*)p;
  return OK;
}
int cudaHostAlloc(void** p, size_t n, unsigned f) { (void)f; *p = calloc(1, n); return *p ? OK : fail(E_NOMEM); }
int cudaFreeHost(void* p) { free(p); return OK; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int kind, void* st) {
  note("copy %d %p %p %zu %p", kind, d, (void*)s, n, st);
  if (kind == 1 || kind == 2) memcpy(d, s, n);
  return OK;
}
int cudaMemcpy(void* d, const void* s, size_t n, int kind) { return cudaMemcpyAsync(d, s, n, kind, NULL); }
int cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, int kind, void* st) {
  note("copy2d %d %p %zu %p %zu %zu %zu %p", kind, d, dp, (void*)s, sp, w, h, st);
  return OK;
}
int cudaMemsetAsync(void* d, int v, size_t n, void* st) { note("memset %p %d %zu %p", d, v, n, st); return OK; }

/* ---- launches ---- */
static struct { const void* fun; char name[224]; } funs[8192];
static int nfuns;
void** __cudaRegisterFatBinary(void* b) { static void* h; (void)b; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterFunction(void** h, const char* fun, char* dfun, const char* name, int lim, void* a,
                            void* b, void* c, void* d, int* e) {
  (void)h; (void)dfun; (void)lim; (void)a; (void)b; (void)c; (void)d; (void)e;
  if (nfuns < 8192) {
    funs[nfuns].fun = fun;
    snprintf(funs[nfuns++].name, sizeof funs[0].name, "%s", name);
  }
}
void __cudaRegisterVar(void** h, char* v, char* a, const char* n, int ext, size_t s, int c, int g) {
  (void)h; (void)v; (void)a; (void)n; (void)ext; (void)s; (void)c; (void)g;
}
static int launch(const void* fun, dim3 g, dim3 b, size_t smem, void* st) {
  const char* name = "?";
  for (int i = 0; i < nfuns; ++i)
    if (funs[i].fun == fun) name = funs[i].name;
  note("launch %s %u %u %u %u %zu %p%s", name, g.x, g.y, g.z, b.x * b.y * b.z, smem, st,
       st && st == capturing ? " captured" : "");
  if (!g.x || !g.y || !g.z || g.x > 2147483647u || g.y > 65535 || g.z > 65535 || !b.x || !b.y || !b.z ||
      b.x > 1024 || b.y > 1024 || b.z > 64 || (uint64_t)b.x * b.y * b.z > 1024)
    return fail(E_CONFIG);
  return OK;
}
static struct { dim3 g, b; size_t smem; void* st; } pending;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void* st) {
  pending.g = g; pending.b = b; pending.smem = smem; pending.st = st;
  return 0;
}
int __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  *g = pending.g; *b = pending.b; *smem = pending.smem; *(void**)st = pending.st;
  return OK;
}
int __cudaGetKernel(void** k, const void* fun) { *k = (void*)fun; return OK; }
int __cudaLaunchKernel(void* k, dim3 g, dim3 b, void** args, size_t smem, void* st) { (void)args; return launch(k, g, b, smem, st); }
int cudaLaunchCooperativeKernel(const void* f, dim3 g, dim3 b, void** args, size_t smem, void* st) { (void)args; return launch(f, g, b, smem, st); }
typedef struct { dim3 g, b; size_t smem; void* st; } LaunchConfig;
int cudaLaunchKernelExC(const LaunchConfig* c, const void* f, void** args) { (void)args; return launch(f, c->g, c->b, c->smem, c->st); }
int cudaFuncSetAttribute(const void* f, int a, int v) { (void)f; (void)a; (void)v; return OK; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int b, size_t s, unsigned fl) {
  (void)f; (void)b; (void)s; (void)fl; *n = 2; return OK;
}

/* ---- device, streams, events, graphs ---- */
int cudaGetDevice(int* d) { *d = 0; return OK; }
int cudaSetDevice(int d) { return d == 0 ? OK : fail(101); }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)d; *v = a == 16 ? 152 : a == 38 ? 129 << 20 : 0; return OK; }
int cudaGetLastError(void) { const int e = last_error; last_error = OK; return e; }
const char* cudaGetErrorString(int e) { static char s[32]; snprintf(s, sizeof s, "error %d", e); return s; }
int cudaGetSymbolAddress(void** p, const void* s) { (void)s; *p = NULL; return fail(E_VALUE); }
int cudaStreamCreateWithFlags(void** s, unsigned f) { (void)f; *s = malloc(8); return OK; }
int cudaStreamDestroy(void* s) { free(s); return OK; }
int cudaStreamSynchronize(void* s) { note("sync %p", s); return s && s == capturing ? fail(900) : OK; }
int cudaStreamWaitEvent(void* s, void* e, unsigned f) { (void)s; (void)e; (void)f; return OK; }
int cudaStreamIsCapturing(void* s, int* c) { *c = s && s == capturing; return OK; }
int cudaStreamBeginCapture(void* s, int m) { (void)m; note("capture %p", s); capturing = s; return OK; }
int cudaStreamEndCapture(void* s, void** g) { note("endcapture %p", s); capturing = NULL; *g = malloc(8); return OK; }
int cudaGraphInstantiate(void** e, void* g, unsigned long long f) { (void)g; (void)f; *e = malloc(8); return OK; }
int cudaGraphLaunch(void* e, void* s) { note("graph %p %p", e, s); return OK; }
int cudaGraphDestroy(void* g) { free(g); return OK; }
int cudaGraphExecDestroy(void* e) { free(e); return OK; }
int cudaEventCreate(void** e) { *e = malloc(8); return OK; }
int cudaEventCreateWithFlags(void** e, unsigned f) { (void)f; *e = malloc(8); return OK; }
int cudaEventDestroy(void* e) { free(e); return OK; }
int cudaEventRecord(void* e, void* s) { (void)e; (void)s; return OK; }
int cudaEventSynchronize(void* e) { (void)e; return OK; }
int cudaEventElapsedTime(float* t, void* a, void* b) { (void)a; (void)b; *t = 1.f; return OK; }

/* ---- cuBLAS and cuSOLVER: handles and work sizes; the routines do nothing ---- */
int cublasCreate_v2(void** h) { *h = malloc(8); return 0; }
int cublasDestroy_v2(void* h) { free(h); return 0; }
int cublasSetStream_v2(void) { return 0; }
int cublasSetMathMode(void) { return 0; }
int cublasDgemm_v2(void) { note("cublasDgemm"); return 0; }
int cublasDsyrk_v2(void) { note("cublasDsyrk"); return 0; }
int cublasDtrsm_v2(void) { return 0; }
int cusolverDnCreate(void** h) { *h = malloc(8); return 0; }
int cusolverDnDestroy(void* h) { free(h); return 0; }
int cusolverDnSetStream(void) { return 0; }
int cusolverDnDpotrf_bufferSize(void* h, int u, int n, void* a, int lda, int* lw) {
  (void)h; (void)u; (void)n; (void)a; (void)lda; *lw = 64; return 0;
}
int cusolverDnDsyevd_bufferSize(void* h, int j, int u, int n, void* a, int lda, void* w, int* lw) {
  (void)h; (void)j; (void)u; (void)n; (void)a; (void)lda; (void)w; *lw = 64; return 0;
}
int cusolverDnDpotrf(void) { return 0; }
int cusolverDnDsyevd(void) { return 0; }
