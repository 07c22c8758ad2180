/* A CUDA runtime without a device, for tests of the library's host logic: device memory is
 * host memory, kernels do not run but are recorded (name and grid), and the n-th cudaMalloc
 * from now on can be made to fail.  Linked with the library's objects in place of libcudart. */
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3;
typedef struct { dim3 grid, block; size_t smem; void *stream, *attrs; unsigned n; } launch_config;

enum { MOST = 4096 };
static struct { const void *fun; const char *name; } kernels[MOST];
static int n_kernels, fail_in, n_launches;
static struct { const char *name; dim3 grid; } launches[MOST];
static dim3 pushed_grid, pushed_block;

/* what the tests drive and read */
void fake_fail_malloc(int nth) { fail_in = nth; }
int fake_launches(void) { return n_launches; }
const char *fake_launch_name(int k) { return launches[k].name; }
unsigned fake_launch_grid(int k, int axis) { return axis == 0 ? launches[k].grid.x : axis == 1 ? launches[k].grid.y : launches[k].grid.z; }

static int launch(const void *fun, dim3 grid, void **args) {
  const char *name = "";
  for (int k = 0; k < n_kernels; ++k)
    if (kernels[k].fun == fun) name = kernels[k].name;
  if (n_launches < MOST) {
    launches[n_launches].name = name;
    launches[n_launches++].grid = grid;
  }
  if (strstr(name, "k_classify") && *(int *)args[4] == 0) { /* 64 sites next to solid ones in 4 warps */
    unsigned *count = *(unsigned **)args[3];
    count[0] = 64;
    count[1] = 4;
  }
  return 0;
}

void **__cudaRegisterFatBinary(void *b) { (void)b; static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterVar(void **h, char *a, char *b, const char *c, int d, size_t e, int f, int g) { (void)h; (void)a; (void)b; (void)c; (void)d; (void)e; (void)f; (void)g; }
void __cudaRegisterFunction(void **h, const char *fun, char *dev, const char *name, int a, void *b, void *c, void *d, void *e, int *f) {
  (void)h; (void)dev; (void)a; (void)b; (void)c; (void)d; (void)e; (void)f;
  if (n_kernels < MOST) {
    kernels[n_kernels].fun = fun;
    kernels[n_kernels++].name = name;
  }
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void *st) { (void)s; (void)st; pushed_grid = g; pushed_block = b; return 0; }
int __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *st) { *g = pushed_grid; *b = pushed_block; *s = 0; *(void **)st = 0; return 0; }
int __cudaGetKernel(const void **k, const void *fun) { *k = fun; return 0; }
int __cudaLaunchKernel(const void *k, dim3 g, dim3 b, void **args, size_t s, void *st) { (void)b; (void)s; (void)st; return launch(k, g, args); }
int cudaLaunchKernelExC(const launch_config *c, const void *fun, void **args) { return launch(fun, c->grid, args); }

static int take(void **p, size_t n) {
  if (fail_in && --fail_in == 0) return 2; /* cudaErrorMemoryAllocation */
  return (*p = calloc(1, n ? n : 1)) ? 0 : 2;
}
int cudaMalloc(void **p, size_t n) { return take(p, n); }
int cudaMallocAsync(void **p, size_t n, void *st) { (void)st; return take(p, n); }
int cudaHostAlloc(void **p, size_t n, unsigned f) { (void)f; return (*p = calloc(1, n)) ? 0 : 2; }
int cudaFree(void *p) { free(p); return 0; }
int cudaFreeAsync(void *p, void *st) { (void)st; free(p); return 0; }
int cudaFreeHost(void *p) { free(p); return 0; }
int cudaMemcpy(void *d, const void *s, size_t n, int k) { (void)k; if (!d || !s) return 1; memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *st) { (void)st; return cudaMemcpy(d, s, n, k); }
int cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, int k, void *st) {
  (void)k; (void)st;
  for (size_t r = 0; r < h; ++r) memcpy((char *)d + r * dp, (const char *)s + r * sp, w);
  return 0;
}
int cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return 0; }
int cudaMemsetAsync(void *d, int v, size_t n, void *st) { (void)st; memset(d, v, n); return 0; }
int cudaDeviceGetAttribute(int *v, int a, int d) { (void)a; (void)d; *v = 152; return 0; }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaSetDevice(int d) { (void)d; return 0; }
int cudaGetLastError(void) { return 0; }
const char *cudaGetErrorString(int e) { (void)e; return "fake error"; }
int cudaPointerGetAttributes(void *a, const void *p) { (void)a; (void)p; return 1; } /* pageable host memory */
int cudaFuncSetAttribute(const void *f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, size_t s, unsigned fl) { (void)f; (void)b; (void)s; (void)fl; *n = 1; return 0; }
int cudaGetDriverEntryPointByVersion(const char *s, void **p, unsigned v, unsigned long long f, void *q) { (void)s; (void)v; (void)f; (void)q; *p = 0; return 1; }
int cudaGetSymbolAddress(void **p, const void *s) { (void)s; *p = 0; return 1; }
int cudaStreamCreate(void **s) { *s = (void *)1; return 0; }
int cudaStreamDestroy(void *s) { (void)s; return 0; }
int cudaStreamSynchronize(void *s) { (void)s; return 0; }
int cudaStreamBeginCapture(void *s, int m) { (void)s; (void)m; return 1; }
int cudaStreamEndCapture(void *s, void **g) { (void)s; (void)g; return 1; }
int cudaGraphInstantiate(void **e, void *g, unsigned long long f) { (void)e; (void)g; (void)f; return 1; }
int cudaGraphLaunch(void *e, void *s) { (void)e; (void)s; return 1; }
int cudaGraphDestroy(void *g) { (void)g; return 0; }
int cudaGraphExecDestroy(void *e) { (void)e; return 0; }
int cudaEventCreate(void **e) { *e = (void *)1; return 0; }
int cudaEventCreateWithFlags(void **e, unsigned f) { (void)f; *e = (void *)1; return 0; }
int cudaEventDestroy(void *e) { (void)e; return 0; }
int cudaEventRecord(void *e, void *s) { (void)e; (void)s; return 0; }
int cudaEventSynchronize(void *e) { (void)e; return 0; }
int cudaEventElapsedTime(float *t, void *a, void *b) { (void)a; (void)b; *t = 0; return 0; }
