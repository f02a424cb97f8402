/* A CUDA runtime of the host alone, preloaded in front of the real one: device
 * memory is host memory, kernels do nothing, and every launch, copy, event
 * record and wait is logged in order.  The fake_fail-th launch fails. */
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3_;
typedef struct { dim3_ grid, block; size_t smem; void *stream; } config_;

int fake_fail = 0;
static int launches = 0, last = 0;
static long handles = 0x1000;
static char text[1 << 16];
static size_t len = 0;

static int put(const char *what, const void *a, const void *b) {
    len += (size_t)snprintf(text + len, sizeof text - len, "%s %ld %ld\n", what, (long)a, (long)b);
    return 0;
}
const char *fake_log(void) { return text; }
void fake_reset(int fail) { fake_fail = fail, launches = 0, len = 0, text[0] = 0, last = 0; }
static int launch(void *stream) {
    if (++launches == fake_fail) return last = 719;
    return put("launch", stream, 0);
}

void **__cudaRegisterFatBinary(void *f) { static void *h; (void)f; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *f, char *n, const char *d, int t, void *a, void *b, void *c, void *e, int *w) {
    (void)h, (void)f, (void)n, (void)d, (void)t, (void)a, (void)b, (void)c, (void)e, (void)w;
}
void __cudaRegisterVar(void **h, char *v, char *a, const char *n, int e, size_t s, int c, int g) {
    (void)h, (void)v, (void)a, (void)n, (void)e, (void)s, (void)c, (void)g;
}
static config_ pushed;
unsigned __cudaPushCallConfiguration(dim3_ g, dim3_ b, size_t m, void *s) { pushed = (config_){g, b, m, s}; return 0; }
int __cudaPopCallConfiguration(dim3_ *g, dim3_ *b, size_t *m, void **s) {
    *g = pushed.grid, *b = pushed.block, *m = pushed.smem, *s = pushed.stream;
    return 0;
}
int __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return 0; }
int __cudaLaunchKernel(void *f, dim3_ g, dim3_ b, void **a, size_t m, void *s) { (void)f, (void)g, (void)b, (void)a, (void)m; return launch(s); }
int cudaLaunchKernelExC(const config_ *c, const void *f, void **a) { (void)f, (void)a; return launch(c->stream); }

int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int *v, int a, int d) { (void)a, (void)d; *v = 152; return 0; }
int cudaDeviceGetStreamPriorityRange(int *l, int *h) { *l = 0, *h = -5; return 0; }
int cudaDeviceSynchronize(void) { return 0; }
int cudaGetLastError(void) { int e = last; last = 0; return e; }
int cudaFuncSetAttribute(const void *f, int a, int v) { (void)f, (void)a, (void)v; return 0; }
int cudaGetSymbolAddress(void **p, const void *s) { static char room[1 << 16]; (void)s; *p = room; return 0; }
int cudaMalloc(void **p, size_t n) { return posix_memalign(p, 256, n ? n : 1) ? 2 : 0; }
int cudaFree(void *p) { free(p); return 0; }
static char sum[40];
const char *fake_last_upload(void) { return sum; }  /* bytes and a checksum */
int cudaMemcpy(void *d, const void *s, size_t n, int k) {
    unsigned long long h = 1469598103934665603ull;
    (void)k;
    memcpy(d, s, n);
    for (size_t i = 0; i < n; ++i) h = (h ^ ((const unsigned char *)s)[i]) * 1099511628211ull;
    snprintf(sum, sizeof sum, "%zu:%llx", n, h);
    return 0;
}
int cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *t) { (void)d, (void)s, (void)n, (void)k; return put("copy", t, 0); }
int cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, int k, void *t) {
    (void)d, (void)dp, (void)s, (void)sp, (void)w, (void)h, (void)k;
    return put("copy", t, 0);
}
int cudaMemsetAsync(void *d, int v, size_t n, void *t) { (void)d, (void)v, (void)n; return put("copy", t, 0); }
int cudaStreamCreateWithFlags(void **s, unsigned f) { (void)f; *s = (void *)(handles += 16); return 0; }
int cudaStreamCreateWithPriority(void **s, unsigned f, int p) { (void)p; return cudaStreamCreateWithFlags(s, f); }
int cudaStreamDestroy(void *s) { (void)s; return 0; }
int cudaStreamSynchronize(void *s) { (void)s; return 0; }
int cudaStreamGetId(void *s, unsigned long long *id) { *id = (unsigned long long)(size_t)s + 1; return 0; }
int cudaThreadExchangeStreamCaptureMode(int *m) { (void)m; return 0; }
int cudaEventCreateWithFlags(void **e, unsigned f) { return cudaStreamCreateWithFlags(e, f); }
int cudaEventDestroy(void *e) { (void)e; return 0; }
int cudaEventQuery(void *e) { (void)e; return 0; }
int cudaEventRecord(void *e, void *s) { return put("record", e, s); }
int cudaStreamWaitEvent(void *s, void *e, unsigned f) { (void)f; return put("wait", s, e); }
int cudaStreamGetCaptureInfo(void *s, int *st, unsigned long long *id) { (void)s; *st = 0; if (id) *id = 0; return 0; }
