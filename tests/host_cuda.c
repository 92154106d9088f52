/* A CUDA runtime for tests of the library's host code on a machine without a GPU: device
 * memory is host memory, copies and fills happen at once, streams and events are names, and
 * a kernel launch runs `on_launch` (set by the test, which plays the kernel's part where the
 * host waits for its words) instead of a kernel.  Every call is counted; a test can make an
 * allocation or a launch fail, and name the current device. */
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

typedef struct { uint32_t x, y, z; } dim3_;
enum { OK = 0, NO_MEMORY = 2, LAUNCH_FAILED = 719 };

/* what a test sets and reads */
void (*host_on_launch)(const char *name, void **args) = 0;
int host_fail_malloc = 0;  /* fail the allocation so many calls ahead (1: the next) */
int host_fail_launch = 0;  /* the same of launches (cudaGetLastError tells) */
int host_device = 0, host_devices = 1;
size_t host_malloc_max = 0; /* the largest allocation of device memory */
size_t host_new_max = 0;   /* the largest piece of host memory that the library took by `new` */
uint64_t host_mallocs = 0, host_attributes = 0, host_stream_uploads = 0, host_plain_uploads = 0;
size_t host_bytes = 0;     /* device memory held */
size_t host_total = (size_t)256 << 30;
static int last_error = OK;

void *__wrap__Znwm(size_t n) {
    if (n > host_new_max) host_new_max = n;
    return malloc(n ? n : 1);
}

/* kernels by the address of their stub */
static struct { const void *stub; const char *name; } fn[8192];
static int n_fn = 0;
static const char *name_of(const void *stub) {
    for (int i = 0; i < n_fn; ++i)
        if (fn[i].stub == stub) return fn[i].name;
    return "?";
}
void **__cudaRegisterFatBinary(void *f) { static void *h; (void)f; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *stub, char *dev, const char *name, int lim, void *a,
                            void *b, void *c, void *d, int *w) {
    (void)h, (void)dev, (void)lim, (void)a, (void)b, (void)c, (void)d, (void)w;
    if (n_fn < 8192) fn[n_fn].stub = stub, fn[n_fn++].name = name;
}
void __cudaRegisterVar(void **h, char *v, char *dev, const char *name, int e, size_t s, int c, int g) {
    (void)h, (void)v, (void)dev, (void)name, (void)e, (void)s, (void)c, (void)g;
}
static __thread struct { dim3_ grid, block; size_t smem; void *stream; } call;
unsigned __cudaPushCallConfiguration(dim3_ g, dim3_ b, size_t smem, void *st) {
    call.grid = g, call.block = b, call.smem = smem, call.stream = st;
    return 0;
}
int __cudaPopCallConfiguration(dim3_ *g, dim3_ *b, size_t *smem, void **st) {
    *g = call.grid, *b = call.block, *smem = call.smem, *st = call.stream;
    return OK;
}
int __cudaGetKernel(const void **k, const void *stub) { return *k = stub, OK; }
int __cudaLaunchKernel(const void *k, dim3_ g, dim3_ b, void **args, size_t smem, void *st) {
    (void)g, (void)b, (void)smem, (void)st;
    if (host_fail_launch > 0 && --host_fail_launch == 0) return last_error = LAUNCH_FAILED;
    if (host_on_launch) host_on_launch(name_of(k), args);
    return OK;
}
int cudaGetLastError(void) { int e = last_error; return last_error = OK, e; }
const char *cudaGetErrorString(int e) { return e == OK ? "ok" : "error"; }

/* memory */
static int take(void **p, size_t n) {
    size_t *b = calloc(1, n + 64);
    if (!b) return NO_MEMORY;
    *b = n, host_bytes += n, *p = (char *)b + 64;
    return OK;
}
int cudaMalloc(void **p, size_t n) {
    ++host_mallocs;
    if (n > host_malloc_max) host_malloc_max = n;
    if (host_fail_malloc > 0 && --host_fail_malloc == 0) return last_error = NO_MEMORY;
    return take(p, n);
}
int cudaFree(void *p) {
    if (!p) return OK;
    size_t *b = (size_t *)((char *)p - 64);
    host_bytes -= *b;
    free(b);
    return OK;
}
int cudaMallocHost(void **p, size_t n) { return *p = calloc(1, n), *p ? OK : NO_MEMORY; }
int cudaHostAlloc(void **p, size_t n, unsigned f) { return (void)f, cudaMallocHost(p, n); }
int cudaFreeHost(void *p) { return free(p), OK; }
int cudaHostGetDevicePointer(void **d, void *h, unsigned f) { return (void)f, *d = h, OK; }
int cudaMemGetInfo(size_t *f, size_t *t) { return *f = host_total - host_bytes, *t = host_total, OK; }
int cudaMemcpy(void *d, const void *s, size_t n, int kind) {
    host_plain_uploads += kind == 1;
    return memcpy(d, s, n), OK;
}
int cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st) {
    (void)st, host_stream_uploads += kind == 1;
    return memcpy(d, s, n), OK;
}
int cudaMemset(void *d, int v, size_t n) { return memset(d, v, n), OK; }
int cudaMemsetAsync(void *d, int v, size_t n, void *st) { return (void)st, memset(d, v, n), OK; }
int cudaGetSymbolAddress(void **p, const void *s) { return *p = (void *)s, OK; }

/* devices, streams, events, graphs */
int cudaGetDeviceCount(int *n) { return *n = host_devices, OK; }
int cudaSetDevice(int d) { return host_device = d, OK; }
int cudaGetDevice(int *d) { return *d = host_device, OK; }
int cudaDeviceGetAttribute(int *v, int a, int d) { return (void)a, (void)d, *v = 152, OK; }
int cudaFuncSetAttribute(const void *f, int a, int v) { return (void)f, (void)a, (void)v, ++host_attributes, OK; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, size_t s, unsigned fl) {
    return (void)f, (void)b, (void)s, (void)fl, *n = 2, OK;
}
static int any;
int cudaStreamCreateWithFlags(void **s, unsigned f) { return (void)f, *s = &any, OK; }
int cudaEventCreate(void **e) { return *e = &any, OK; }
int cudaEventCreateWithFlags(void **e, unsigned f) { return (void)f, *e = &any, OK; }
int cudaEventElapsedTime(float *ms, void *a, void *b) { return (void)a, (void)b, *ms = 1.f, OK; }
int cudaStreamDestroy(void *s) { return (void)s, OK; }
int cudaStreamSynchronize(void *s) { return (void)s, OK; }
int cudaStreamWaitEvent(void *s, void *e, unsigned f) { return (void)s, (void)e, (void)f, OK; }
int cudaStreamBeginCapture(void *s, int m) { return (void)s, (void)m, OK; }
int cudaStreamEndCapture(void *s, void **g) { return (void)s, *g = &any, OK; }
int cudaEventDestroy(void *e) { return (void)e, OK; }
int cudaEventQuery(void *e) { return (void)e, OK; }
int cudaEventRecord(void *e, void *s) { return (void)e, (void)s, OK; }
int cudaEventSynchronize(void *e) { return (void)e, OK; }
int cudaDeviceSynchronize(void) { return OK; }
int cudaGraphDestroy(void *g) { return (void)g, OK; }
int cudaGraphExecDestroy(void *g) { return (void)g, OK; }
int cudaGraphGetNodes(void *g, void **n, size_t *k) { return (void)g, (void)n, *k = 0, OK; }
int cudaGraphInstantiate(void **x, void *g, unsigned long long f) { return (void)g, (void)f, *x = &any, OK; }
int cudaGraphLaunch(void *x, void *s) { return (void)x, (void)s, OK; }
int cudaGraphNodeGetType(void *n, int *t) { return (void)n, *t = 0, OK; }
int cudaGetDriverEntryPointByVersion(const char *n, void **p, unsigned v, unsigned long long f, int *q) {
    return (void)n, (void)v, (void)f, *p = 0, *q = 1, OK;
}
