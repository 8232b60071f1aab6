/* A CUDA runtime without a device, preloaded under liblrugb.so by
 * test_host_paths_cpu.py: memory comes from the host, kernels are not run, and
 * what the library asks for (allocations, launches, function attributes per
 * device) is recorded.  A launch with more dynamic shared memory than its
 * function was allowed on the current device is refused, as the runtime does;
 * allocations and launches can be refused on demand. */
#include <stddef.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3_t;
enum { OK = 0, INVALID = 1, NOMEM = 2, MAXF = 4096, MAXL = 65536, DEVICES = 2 };

static struct { const void* fn; const char* name; int smem[DEVICES]; } funcs[MAXF];
static int nfuncs, device, last;
static struct { int func, device, ok; unsigned grid_x; void* arg; } launches[MAXL];
static int nlaunches;
static size_t alloc_limit = (size_t)-1, total_limit = (size_t)-1, total;
static char refuse[64], watch[64];
static int watch_arg;
static struct { size_t bytes; int ok; void* p; } allocs[MAXL];
static int nallocs, first;

static int fail(int e) { last = e; return e; }

/* ---- what the test reads and sets ---- */
void fake_alloc_limit(size_t b) { alloc_limit = b; }      /* of one allocation */
void fake_total_limit(size_t b) { total_limit = b; }      /* of all together */
void fake_refuse_launch(const char* s) { strncpy(refuse, s, sizeof refuse - 1); }
void fake_watch(const char* s, int arg) { strncpy(watch, s, sizeof watch - 1); watch_arg = arg; }
void fake_reset(void) { nlaunches = 0; first = nallocs; }
int fake_launches(void) { return nlaunches; }
const char* fake_launch_name(int i) { return funcs[launches[i].func].name; }
int fake_launch_ok(int i) { return launches[i].ok; }
unsigned fake_launch_grid(int i) { return launches[i].grid_x; }
void* fake_launch_arg(int i) { return launches[i].arg; }
int fake_allocs(void) { return nallocs - first; }
size_t fake_alloc_bytes(int i) { return allocs[first + i].bytes; }
int fake_alloc_ok(int i) { return allocs[first + i].ok; }

/* ---- registration and launches ---- */
void** __cudaRegisterFatBinary(void* f) { (void)f; return (void**)malloc(8); }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void** h, char* v, char* a, const char* n, int e, size_t s, int c, int g) {
    (void)h; (void)v; (void)a; (void)n; (void)e; (void)s; (void)c; (void)g;
}
void __cudaRegisterFunction(void** h, const char* fn, char* d, const char* name, int t, void* a, void* b, void* c,
                            void* e, int* w) {
    (void)h; (void)d; (void)t; (void)a; (void)b; (void)c; (void)e; (void)w;
    if (nfuncs < MAXF) { funcs[nfuncs].fn = fn; funcs[nfuncs].name = name; ++nfuncs; }
}
static int find(const void* fn) {
    for (int i = 0; i < nfuncs; ++i)
        if (funcs[i].fn == fn) return i;
    return -1;
}
static struct { dim3_t g, b; size_t s; void* st; } cfg;
unsigned __cudaPushCallConfiguration(dim3_t g, dim3_t b, size_t s, void* st) {
    cfg.g = g; cfg.b = b; cfg.s = s; cfg.st = st;
    return 0;
}
int __cudaPopCallConfiguration(dim3_t* g, dim3_t* b, size_t* s, void* st) {
    *g = cfg.g; *b = cfg.b; *s = cfg.s; *(void**)st = cfg.st;
    return OK;
}
int __cudaGetKernel(void** k, const void* fn) { *k = (void*)fn; return OK; }
int __cudaLaunchKernel(void* k, dim3_t g, dim3_t b, void** args, size_t smem, void* st) {
    (void)b; (void)st;
    const int f = find(k);
    if (f < 0) return fail(INVALID);
    int ok = smem <= 48 * 1024 || (int)smem <= funcs[f].smem[device];
    if (refuse[0] && strstr(funcs[f].name, refuse)) ok = 0;
    if (nlaunches < MAXL) {
        launches[nlaunches].func = f;
        launches[nlaunches].device = device;
        launches[nlaunches].ok = ok;
        launches[nlaunches].grid_x = g.x;
        launches[nlaunches].arg = watch[0] && strstr(funcs[f].name, watch) ? *(void**)args[watch_arg] : NULL;
        ++nlaunches;
    }
    return ok ? OK : fail(INVALID);
}
int cudaFuncSetAttribute(const void* fn, int attr, int value) {
    const int f = find(fn);
    if (f < 0) return fail(INVALID);
    if (attr == 8) funcs[f].smem[device] = value;   /* MaxDynamicSharedMemorySize */
    return OK;
}

/* ---- memory ---- */
static int alloc(void** p, size_t n) {
    int ok = n <= alloc_limit && total + n <= total_limit;
    *p = ok ? aligned_alloc(256, (n + 255) / 256 * 256) : NULL;   /* untouched pages cost nothing */
    ok = *p != NULL;
    if (ok) total += n;
    if (nallocs < MAXL) { allocs[nallocs].bytes = n; allocs[nallocs].ok = ok; allocs[nallocs].p = *p; ++nallocs; }
    return ok ? OK : fail(NOMEM);
}
static int release(void* p) {
    for (int i = 0; p && i < nallocs; ++i)
        if (allocs[i].p == p) { total -= allocs[i].bytes; allocs[i].p = NULL; }
    free(p);
    return OK;
}
int cudaMalloc(void** p, size_t n) { return alloc(p, n); }
int cudaMallocAsync(void** p, size_t n, void* s) { (void)s; return alloc(p, n); }
int cudaFree(void* p) { return release(p); }
int cudaFreeAsync(void* p, void* s) { (void)s; return release(p); }
int cudaMemcpy(void* d, const void* s, size_t n, int k) { (void)k; memcpy(d, s, n); return OK; }
int cudaMemcpyAsync(void* d, const void* s, size_t n, int k, void* st) { (void)d; (void)s; (void)n; (void)k; (void)st; return OK; }
int cudaMemset(void* d, int v, size_t n) { (void)d; (void)v; (void)n; return OK; }
int cudaMemsetAsync(void* d, int v, size_t n, void* st) { (void)d; (void)v; (void)n; (void)st; return OK; }

/* ---- devices, streams, events ---- */
int cudaSetDevice(int d) { if (d < 0 || d >= DEVICES) return fail(101); device = d; return OK; }
int cudaGetDevice(int* d) { *d = device; return OK; }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)a; (void)d; *v = 152; return OK; }
int cudaDeviceSynchronize(void) { return OK; }
int cudaStreamSynchronize(void* s) { (void)s; return OK; }
int cudaStreamIsCapturing(void* s, int* st) { (void)s; *st = 0; return OK; }
int cudaGetLastError(void) { const int e = last; last = OK; return e; }
int cudaPeekAtLastError(void) { return last; }
int cudaEventCreate(void** e) { *e = malloc(1); return OK; }
int cudaEventDestroy(void* e) { free(e); return OK; }
int cudaEventRecord(void* e, void* s) { (void)e; (void)s; return OK; }
int cudaEventElapsedTime(float* t, void* a, void* b) { (void)a; (void)b; *t = 0; return OK; }
int cudaGetSymbolAddress(void** p, const void* s) { (void)s; *p = malloc(256); return OK; }
static int encode_tiled(void) { return 0; }
int cudaGetDriverEntryPointByVersion(const char* s, void** p, unsigned v, unsigned long long f, int* q) {
    (void)s; (void)v; (void)f;
    *p = (void*)encode_tiled;
    *q = 0;
    return OK;
}
