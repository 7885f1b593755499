/* A stand-in for the CUDA runtime on a machine without a GPU: the host code of libtn.so plans,
 * allocates, captures and launches as usual, device memory is host memory and kernels do nothing.
 * It counts the calls of each function and can make the next call of one fail. */
#include <stddef.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>

enum { kCounters = 64, kNone = 0, kInvalidValue = 1, kOutOfMemory = 2 };
static struct {
    const char *name;
    long calls, ok, fail;  /* `fail` calls fail after `ok` more calls */
} counters[kCounters];

static int call(const char *name) {
    int i = 0;
    while (i < kCounters && counters[i].name && strcmp(counters[i].name, name)) ++i;
    if (i == kCounters) abort();
    counters[i].name = name;
    counters[i].calls++;
    if (counters[i].fail == 0) return kNone;
    if (counters[i].ok > 0) {
        counters[i].ok--;
        return kNone;
    }
    counters[i].fail--;
    return kOutOfMemory;
}
static int last_error;
static int status(const char *name) {
    const int e = call(name);
    if (e) last_error = e;
    return e;
}
long fake_calls(const char *name) {
    for (int i = 0; i < kCounters && counters[i].name; ++i)
        if (!strcmp(counters[i].name, name)) return counters[i].calls;
    return 0;
}
void fake_fail(const char *name, long ok, long fail) {
    const int before = (int)fake_calls(name);
    char *copy = strdup(name);
    (void)call(copy);
    for (int i = 0; i < kCounters && counters[i].name; ++i)
        if (!strcmp(counters[i].name, name)) {
            counters[i].calls = before;
            counters[i].ok = ok;
            counters[i].fail = fail;
        }
}

/* objects alive: memory blocks, streams, events, graphs, executable graphs */
static long alive[5];
long fake_alive(int kind) { return alive[kind]; }
static void *object(int kind) {
    alive[kind]++;
    return malloc(16);
}
static int drop(const char *name, int kind, void *p) {
    alive[kind]--;
    free(p);
    return status(name);
}

int cudaMalloc(void **p, size_t n) {
    const int e = status("cudaMalloc");
    if (e) return e;
    size_t *m = mmap(NULL, n + 4096, PROT_READ | PROT_WRITE,
                     MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (m == MAP_FAILED) return last_error = kOutOfMemory;
    *m = n + 4096;
    *p = (char *)m + 4096;
    alive[0]++;
    return kNone;
}
int cudaFree(void *p) {
    if (p) {
        size_t *m = (size_t *)((char *)p - 4096);
        munmap(m, *m);
        alive[0]--;
    }
    return status("cudaFree");
}
int cudaMemGetInfo(size_t *f, size_t *t) {
    *f = *t = (size_t)200 << 30;
    return status("cudaMemGetInfo");
}
int cudaMemcpy(void *d, const void *s, size_t n, int kind) {
    (void)kind;
    memcpy(d, s, n);
    return status("cudaMemcpy");
}
int cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st) {
    (void)kind, (void)st;
    memcpy(d, s, n);
    return status("cudaMemcpyAsync");
}
int cudaMemsetAsync(void *d, int v, size_t n, void *st) {
    (void)st;
    memset(d, v, n);
    return status("cudaMemsetAsync");
}
int cudaMemcpyFromSymbol(void *d, const void *sym, size_t n, size_t off, int kind) {
    (void)sym, (void)off, (void)kind;
    memset(d, 0, n);
    return status("cudaMemcpyFromSymbol");
}
int cudaMemcpyToSymbol(const void *sym, const void *s, size_t n, size_t off, int kind) {
    (void)sym, (void)s, (void)n, (void)off, (void)kind;
    return status("cudaMemcpyToSymbol");
}
int cudaGetSymbolAddress(void **p, const void *sym) {
    static char scratch[1 << 16];
    (void)sym;
    *p = scratch;
    return status("cudaGetSymbolAddress");
}

int cudaGetDevice(int *d) { return *d = 0, status("cudaGetDevice"); }
int cudaSetDevice(int d) { return (void)d, status("cudaSetDevice"); }
int cudaDeviceGetAttribute(int *v, int attr, int dev) {
    (void)dev;
    *v = attr == 75 ? 10 : attr == 16 ? 152 : 0; /* compute capability 10.x, 152 SMs */
    return status("cudaDeviceGetAttribute");
}
int cudaFuncGetAttributes(void *a, const void *f) { return (void)a, (void)f, status("cudaFuncGetAttributes"); }
int cudaFuncSetAttribute(const void *f, int a, int v) { return (void)f, (void)a, (void)v, status("cudaFuncSetAttribute"); }
int cudaGetLastError(void) {
    const int e = last_error;
    last_error = kNone;
    return e;
}
int cudaPeekAtLastError(void) { return last_error; }
const char *cudaGetErrorString(int e) { return e == kOutOfMemory ? "out of memory" : "error"; }
static int encode_tiled(void) { return 0; }
int cudaGetDriverEntryPointByVersion(const char *name, void **fn, unsigned v, unsigned long long f,
                                     int *result) {
    (void)name, (void)v, (void)f;
    *fn = (void *)encode_tiled;
    if (result) *result = 0;
    return status("cudaGetDriverEntryPointByVersion");
}

int cudaStreamCreateWithFlags(void **s, unsigned f) {
    (void)f;
    const int e = status("cudaStreamCreateWithFlags");
    if (!e) *s = object(1);
    return e;
}
int cudaStreamDestroy(void *s) { return drop("cudaStreamDestroy", 1, s); }
int cudaStreamSynchronize(void *s) { return (void)s, status("cudaStreamSynchronize"); }
int cudaStreamWaitEvent(void *s, void *e, unsigned f) { return (void)s, (void)e, (void)f, status("cudaStreamWaitEvent"); }
int cudaEventCreateWithFlags(void **e, unsigned f) {
    (void)f;
    const int r = status("cudaEventCreateWithFlags");
    if (!r) *e = object(2);
    return r;
}
int cudaEventCreate(void **e) { return cudaEventCreateWithFlags(e, 0); }
int cudaEventDestroy(void *e) { return drop("cudaEventDestroy", 2, e); }
int cudaEventRecord(void *e, void *s) { return (void)e, (void)s, status("cudaEventRecord"); }
int cudaEventSynchronize(void *e) { return (void)e, status("cudaEventSynchronize"); }
int cudaEventElapsedTime(float *ms, void *a, void *b) {
    (void)a, (void)b;
    *ms = 1.f;
    return status("cudaEventElapsedTime");
}

/* capture: `captured` is the stream between begin and end; fake_capture marks one as the caller's */
static void *captured, *callers;
void fake_capture(void *s) { callers = s; }
int cudaStreamBeginCapture(void *s, int mode) {
    (void)mode;
    const int e = status("cudaStreamBeginCapture");
    if (!e) captured = s;
    return e;
}
int cudaStreamEndCapture(void *s, void **g) {
    *g = NULL;
    if (s != captured) return last_error = kInvalidValue;
    captured = NULL;
    const int e = status("cudaStreamEndCapture");
    if (!e) *g = object(3);
    return e;
}
int cudaStreamIsCapturing(void *s, int *c) {
    *c = s && (s == captured || s == callers);
    return status("cudaStreamIsCapturing");
}
int cudaGraphInstantiate(void **x, void *g, unsigned long long f) {
    (void)g, (void)f;
    *x = NULL;
    const int e = status("cudaGraphInstantiate");
    if (!e) *x = object(4);
    return e;
}
int cudaGraphDestroy(void *g) { return drop("cudaGraphDestroy", 3, g); }
int cudaGraphExecDestroy(void *x) { return drop("cudaGraphExecDestroy", 4, x); }
int cudaGraphLaunch(void *x, void *s) { return (void)x, (void)s, status("cudaGraphLaunch"); }

/* kernel launches, as nvcc's host code makes them */
typedef struct { unsigned x, y, z; } dims;
int cudaLaunchKernelExC(const void *cfg, const void *f, void **args) { return (void)cfg, (void)f, (void)args, status("launch"); }
unsigned __cudaPushCallConfiguration(dims g, dims b, size_t n, void *s) { return (void)g, (void)b, (void)n, (void)s, 0; }
int __cudaPopCallConfiguration(dims *g, dims *b, size_t *n, void *s) {
    memset(g, 0, sizeof *g);
    memset(b, 0, sizeof *b);
    *n = 0;
    *(void **)s = NULL;
    return kNone;
}
int __cudaGetKernel(void **k, const void *f) { return *k = (void *)f, kNone; }
int __cudaLaunchKernel(void *k, dims g, dims b, void **a, size_t n, void *s) { return (void)k, (void)g, (void)b, (void)a, (void)n, (void)s, status("launch"); }
int cudaLaunchKernel(void *k, dims g, dims b, void **a, size_t n, void *s) { return __cudaLaunchKernel(k, g, b, a, n, s); }
void **__cudaRegisterFatBinary(void *b) { return (void **)b; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void) {}
void __cudaRegisterVar(void) {}
