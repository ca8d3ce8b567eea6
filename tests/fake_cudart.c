/* A stand-in for the CUDA runtime, preloaded into a test's process, so that
 * the library's host code runs without a GPU: device memory is host memory
 * (counted), kernel launches do nothing (their configurations are recorded),
 * and one launch can be made to fail. */
#include <stddef.h>
#include <stdlib.h>
#include <string.h>

typedef int err_t;
typedef void* ptr_t;
typedef struct { unsigned x, y, z; } dim_t;
typedef struct { dim_t grid, block; size_t smem; ptr_t stream; void* attrs; unsigned n; } config_t;

enum { kMax = 4096, kFailed = 9 /* cudaErrorInvalidConfiguration */ };

/* what a test sets and reads */
int fake_sms = 152, fake_occupancy = 4;
int fake_fail_at = -1;              /* number of the launch that fails */
int fake_launches = 0;
unsigned fake_grid[kMax], fake_block[kMax];
size_t fake_smem[kMax];
size_t fake_bytes = 0, fake_peak = 0; /* allocated now, and at most so far */

static err_t last = 0;
static int handles = 0;

static err_t launched(dim_t g, dim_t b, size_t smem) {
  const int k = fake_launches++;
  if (k < kMax) fake_grid[k] = g.x, fake_block[k] = b.x, fake_smem[k] = smem;
  return k == fake_fail_at ? (last = kFailed) : 0;
}
static ptr_t handle(void) { return (ptr_t)(size_t)(16 + 16 * ++handles); }

/* memory; the size of an allocation stands in front of it */
err_t cudaMalloc(void** p, size_t n) {
  size_t* m = calloc(1, n + 64);
  if (!m) return 2;
  m[0] = n;
  *p = (char*)m + 64;
  fake_bytes += n;
  if (fake_bytes > fake_peak) fake_peak = fake_bytes;
  return 0;
}
err_t cudaFree(void* p) {
  if (!p) return 0;
  size_t* m = (size_t*)((char*)p - 64);
  fake_bytes -= m[0];
  free(m);
  return 0;
}
err_t cudaMallocAsync(void** p, size_t n, ptr_t s) { (void)s; return cudaMalloc(p, n); }
err_t cudaFreeAsync(void* p, ptr_t s) { (void)s; return cudaFree(p); }
err_t cudaMemcpy(void* d, const void* s, size_t n, int k) { (void)k; memcpy(d, s, n); return 0; }
err_t cudaMemcpyAsync(void* d, const void* s, size_t n, int k, ptr_t t) { (void)k; (void)t; memcpy(d, s, n); return 0; }
err_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return 0; }
err_t cudaMemsetAsync(void* d, int v, size_t n, ptr_t t) { (void)t; memset(d, v, n); return 0; }
err_t cudaMemGetInfo(size_t* a, size_t* b) { *a = *b = (size_t)1 << 38; return 0; }

/* launches */
static config_t pushed;
unsigned __cudaPushCallConfiguration(dim_t g, dim_t b, size_t smem, ptr_t s) {
  pushed.grid = g, pushed.block = b, pushed.smem = smem, pushed.stream = s;
  return 0;
}
err_t __cudaPopCallConfiguration(dim_t* g, dim_t* b, size_t* smem, void* s) {
  *g = pushed.grid, *b = pushed.block, *smem = pushed.smem, *(ptr_t*)s = pushed.stream;
  return 0;
}
err_t __cudaGetKernel(ptr_t* k, const void* f) { *k = (ptr_t)f; return 0; }
err_t __cudaLaunchKernel(ptr_t k, dim_t g, dim_t b, void** a, size_t smem, ptr_t s) {
  (void)k; (void)a; (void)s;
  return launched(g, b, smem);
}
err_t cudaLaunchKernelExC(const config_t* c, const void* f, void** a) {
  (void)f; (void)a;
  return launched(c->grid, c->block, c->smem);
}
err_t cudaGetLastError(void) { const err_t e = last; last = 0; return e; }
const char* cudaGetErrorString(err_t e) { return e == kFailed ? "launch rejected" : "no error"; }

/* device, streams, events, graphs */
err_t cudaGetDevice(int* d) { *d = 0; return 0; }
err_t cudaDeviceGetAttribute(int* v, int a, int d) { (void)a; (void)d; *v = fake_sms; return 0; }
err_t cudaDeviceGetStreamPriorityRange(int* a, int* b) { *a = 0; *b = -5; return 0; }
err_t cudaFuncSetAttribute(const void* f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
err_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void* f, int b, size_t s) {
  (void)f; (void)b; (void)s;
  *n = fake_occupancy;
  return 0;
}
err_t cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)s; return 0; }
err_t cudaStreamCreateWithFlags(ptr_t* s, unsigned f) { (void)f; *s = handle(); return 0; }
err_t cudaStreamDestroy(ptr_t s) { (void)s; return 0; }
err_t cudaStreamSynchronize(ptr_t s) { (void)s; return 0; }
err_t cudaStreamWaitEvent(ptr_t s, ptr_t e, unsigned f) { (void)s; (void)e; (void)f; return 0; }
err_t cudaEventCreate(ptr_t* e) { *e = handle(); return 0; }
err_t cudaEventCreateWithFlags(ptr_t* e, unsigned f) { (void)f; *e = handle(); return 0; }
err_t cudaEventDestroy(ptr_t e) { (void)e; return 0; }
err_t cudaEventRecord(ptr_t e, ptr_t s) { (void)e; (void)s; return 0; }
err_t cudaEventSynchronize(ptr_t e) { (void)e; return 0; }
err_t cudaEventElapsedTime(float* t, ptr_t a, ptr_t b) { (void)a; (void)b; *t = 1.0f; return 0; }
err_t cudaStreamBeginCapture(ptr_t s, int m) { (void)s; (void)m; return 0; }
err_t cudaStreamEndCapture(ptr_t s, ptr_t* g) { (void)s; *g = handle(); return 0; }
err_t cudaGraphGetNodes(ptr_t g, ptr_t* n, size_t* c) { (void)g; (void)n; *c = 0; return 0; }
err_t cudaGraphInstantiate(ptr_t* x, ptr_t g, unsigned long long f) { (void)g; (void)f; *x = handle(); return 0; }
err_t cudaGraphLaunch(ptr_t x, ptr_t s) { (void)x; (void)s; return 0; }
err_t cudaGraphDestroy(ptr_t g) { (void)g; return 0; }
err_t cudaGraphExecDestroy(ptr_t x) { (void)x; return 0; }
