/* A CUDA runtime without a GPU, preloaded in front of libcudart by test_fake_runtime_cpu.py: device
 * memory is host memory, kernels do nothing, and a launch is refused as the real runtime refuses it
 * when its dynamic shared memory is beyond 48 KB and the kernel's attribute has not been set on the
 * current device.  fake_limit bounds the bytes allocated at one time. */
#define _GNU_SOURCE
#include <malloc.h>
#include <stddef.h>
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3_t;
enum { kOk = 0, kInvalid = 1, kNoMemory = 2, kDevs = 4, kFuncs = 4096 };
enum { kAttrDynamicSmem = 8, kDevAttrSms = 16 };

static int g_dev, g_last, g_launches, g_refused;
static size_t g_limit = (size_t)8 << 30, g_used;
static const void *g_func[kFuncs];
static int g_attr[kDevs][kFuncs], g_nfunc;

void fake_set_device(int d) { g_dev = d; }
void fake_set_limit(size_t b) { g_limit = b; }
size_t fake_used(void) { return g_used; }
int fake_launches(void) { return g_launches; }
int fake_refused(void) { return g_refused; }

static int err(int e) { if (e) g_last = e; return e; }
static int slot(const void *f) {
  for (int i = 0; i < g_nfunc; ++i) if (g_func[i] == f) return i;
  g_func[g_nfunc] = f;
  return g_nfunc++;
}
static int launch(const void *f, size_t smem) {
  ++g_launches;
  if (smem <= 48 * 1024 || (size_t)g_attr[g_dev][slot(f)] >= smem) return kOk;
  ++g_refused;
  return err(kInvalid);
}
static int take(void **p, size_t n) {
  *p = NULL;
  if (g_used + n > g_limit) return err(kNoMemory);
  *p = calloc(1, n ? n : 1);
  g_used += malloc_usable_size(*p);
  return kOk;
}
static int give(void *p) {
  if (p) g_used -= malloc_usable_size(p);
  free(p);
  return kOk;
}

int cudaGetDevice(int *d) { *d = g_dev; return kOk; }
int cudaDeviceGetAttribute(int *v, int a, int d) { (void)d; *v = a == kDevAttrSms ? 152 : 1; return kOk; }
int cudaGetLastError(void) { int e = g_last; g_last = 0; return e; }
int cudaFuncSetAttribute(const void *f, int a, int v) {
  if (a == kAttrDynamicSmem) g_attr[g_dev][slot(f)] = v;
  return kOk;
}
int __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return kOk; }
int __cudaLaunchKernel(void *k, dim3_t g, dim3_t b, void **a, size_t smem, void *st) {
  (void)g; (void)b; (void)a; (void)st;
  return launch(k, smem);
}
int cudaLaunchCooperativeKernel(const void *f, dim3_t g, dim3_t b, void **a, size_t smem, void *st) {
  (void)g; (void)b; (void)a; (void)st;
  return launch(f, smem);
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, size_t s, unsigned fl) {
  (void)f; (void)b; (void)s; (void)fl;
  *n = 2;
  return kOk;
}
int cudaMalloc(void **p, size_t n) { return take(p, n); }
int cudaMallocAsync(void **p, size_t n, void *st) { (void)st; return take(p, n); }
int cudaFree(void *p) { return give(p); }
int cudaFreeAsync(void *p, void *st) { (void)st; return give(p); }
int cudaMallocHost(void **p, size_t n) { *p = calloc(1, n ? n : 1); return kOk; }
int cudaHostAlloc(void **p, size_t n, unsigned f) { (void)f; return cudaMallocHost(p, n); }
int cudaFreeHost(void *p) { free(p); return kOk; }
int cudaMemGetInfo(size_t *f, size_t *t) { *f = g_limit - g_used; *t = g_limit; return kOk; }
int cudaMemcpy(void *d, const void *s, size_t n, int k) { (void)k; memcpy(d, s, n); return kOk; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *st) { (void)st; return cudaMemcpy(d, s, n, k); }
int cudaMemsetAsync(void *d, int v, size_t n, void *st) { (void)st; memset(d, v, n); return kOk; }
int cudaStreamCreateWithFlags(void **s, unsigned f) { (void)f; *s = (void *)1; return kOk; }
int cudaStreamDestroy(void *s) { (void)s; return kOk; }
int cudaStreamSynchronize(void *s) { (void)s; return kOk; }
int cudaStreamWaitEvent(void *s, void *e, unsigned f) { (void)s; (void)e; (void)f; return kOk; }
int cudaEventCreate(void **e) { *e = (void *)1; return kOk; }
int cudaEventCreateWithFlags(void **e, unsigned f) { (void)f; return cudaEventCreate(e); }
int cudaEventDestroy(void *e) { (void)e; return kOk; }
int cudaEventRecord(void *e, void *s) { (void)e; (void)s; return kOk; }
int cudaEventSynchronize(void *e) { (void)e; return kOk; }
int cudaEventElapsedTime(float *ms, void *a, void *b) { (void)a; (void)b; *ms = 1.f; return kOk; }
