/* A stand-in for the CUDA runtime on a machine without a GPU: "device" memory is
 * host memory, copies are made, kernels are not run.  Counts what is allocated,
 * fails the n-th allocation on request, and asks a callback for the data of
 * device-to-host copies.  Linked with the library's own objects by
 * test_plan_resources.py. */
#include <stddef.h>
#include <stdlib.h>
#include <string.h>

typedef int err;
typedef struct { unsigned x, y, z; } d3;

static long live, made, fail_at = -1;
static void (*d2h)(void *dst, size_t n);

void fake_reset(long fail) { live = made = 0; fail_at = fail; }
long fake_live(void) { return live; }
long fake_made(void) { return made; }
void fake_d2h(void (*cb)(void *, size_t)) { d2h = cb; }

err cudaMalloc(void **p, size_t n) {
    if (made++ == fail_at) return 2;
    *p = calloc(1, n ? n : 1);
    ++live;
    return *p ? 0 : 2;
}
err cudaFree(void *p) {
    if (p) { free(p); --live; }
    return 0;
}
err cudaMallocAsync(void **p, size_t n, void *s) { (void)s; return cudaMalloc(p, n); }
err cudaFreeAsync(void *p, void *s) { (void)s; return cudaFree(p); }
err cudaMemcpy(void *d, const void *s, size_t n, int kind) {
    if (n) memmove(d, s, n);
    if (kind == 2 && d2h) d2h(d, n);
    return 0;
}
err cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st) { (void)st; return cudaMemcpy(d, s, n, kind); }
err cudaMemsetAsync(void *d, int v, size_t n, void *st) { (void)st; memset(d, v, n); return 0; }

err cudaDeviceGetAttribute(int *v, int a, int d) { (void)a; (void)d; *v = 152; return 0; }
err cudaDeviceSynchronize(void) { return 0; }
err cudaStreamSynchronize(void *s) { (void)s; return 0; }
err cudaStreamBeginCapture(void *s, int m) { (void)s; (void)m; return 0; }
err cudaStreamEndCapture(void *s, void **g) { (void)s; *g = NULL; return 0; }
err cudaGraphInstantiate(void **e, void *g, unsigned long long f) { (void)g; (void)f; *e = NULL; return 0; }
err cudaGraphLaunch(void *e, void *s) { (void)e; (void)s; return 0; }
err cudaGraphDestroy(void *g) { (void)g; return 0; }
err cudaGraphExecDestroy(void *e) { (void)e; return 0; }
err cudaEventCreate(void **e) { *e = NULL; return 0; }
err cudaEventDestroy(void *e) { (void)e; return 0; }
err cudaEventRecord(void *e, void *s) { (void)e; (void)s; return 0; }
err cudaEventSynchronize(void *e) { (void)e; return 0; }
err cudaEventElapsedTime(float *t, void *a, void *b) { (void)a; (void)b; *t = 1.f; return 0; }
err cudaGetDevice(int *d) { *d = 0; return 0; }
err cudaGetLastError(void) { return 0; }
const char *cudaGetErrorString(err e) { return e ? "an error" : "no error"; }
err cudaGetSymbolAddress(void **p, const void *s) { *p = (void *)s; return 0; }
err cudaFuncSetAttribute(const void *f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
err cudaLaunchKernelExC(const void *c, const void *f, void **a) { (void)c; (void)f; (void)a; return 0; }
err __cudaLaunchKernel(void *k, d3 g, d3 b, void **a, size_t m, void *s) { (void)k; (void)g; (void)b; (void)a; (void)m; (void)s; return 0; }
err cudaLaunchKernel(const void *k, d3 g, d3 b, void **a, size_t m, void *s) { (void)k; (void)g; (void)b; (void)a; (void)m; (void)s; return 0; }
err __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return 0; }
unsigned __cudaPushCallConfiguration(d3 g, d3 b, size_t m, void *s) { (void)g; (void)b; (void)m; (void)s; return 0; }
err __cudaPopCallConfiguration(d3 *g, d3 *b, size_t *m, void **s) { memset(g, 0, sizeof(*g)); memset(b, 0, sizeof(*b)); *m = 0; *s = NULL; return 0; }
void **__cudaRegisterFatBinary(void *f) { static void *h; (void)f; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *f, char *d, const char *n, int t, void *a, void *b, void *c, void *e, int *w) { (void)h; (void)f; (void)d; (void)n; (void)t; (void)a; (void)b; (void)c; (void)e; (void)w; }
void __cudaRegisterVar(void **h, char *v, char *d, const char *n, int e, size_t s, int c, int g) { (void)h; (void)v; (void)d; (void)n; (void)e; (void)s; (void)c; (void)g; }
