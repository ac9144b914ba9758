/* A CUDA runtime without a GPU, for tests of the host code: device memory is
 * host memory with a budget, copies and clears happen at once, kernels are not
 * run but noted (name, grid, shared memory, device), and a launch whose shared
 * memory is above what its device was told to allow is refused, as the real
 * runtime refuses it.  Two devices; one thread. */
#include <stdint.h>
#include <stdlib.h>
#include <string.h>
#include <sys/mman.h>

typedef struct { unsigned x, y, z; } dim3_t;
enum { OK = 0, INVALID = 1, NO_MEMORY = 2, DEVICES = 2, FUNCS = 1024, BLOCKS = 1 << 16, EVENTS = 1 << 16 };

static struct { const void *host; const char *name; int smem[DEVICES]; } funcs[FUNCS];
static int n_funcs;
static struct { char *p; size_t n; int dev; } blocks[BLOCKS];
static int n_blocks;
static int device, last_error;
static size_t budget[DEVICES], used[DEVICES];

typedef struct { char kind; int func, device; unsigned grid; size_t smem, bytes; } event_t; /* L launch, F function used otherwise, M malloc */
static event_t events[EVENTS];
static int n_events;
static uint64_t patch_bytes, patch_offset, patch_value;

static int fail(int e) { return last_error = e; }
static void note(char kind, int func, unsigned grid, size_t smem, size_t bytes) {
    if (n_events < EVENTS) events[n_events++] = (event_t){kind, func, device, grid, smem, bytes};
}
static int find(const void *host) {
    for (int i = 0; i < n_funcs; ++i)
        if (funcs[i].host == host) return i;
    return -1;
}

/* what the tests ask */
void fake_budget(int dev, size_t bytes) { budget[dev] = bytes; }
size_t fake_used(int dev) { return used[dev]; }
void fake_clear(void) { n_events = 0; }
int fake_events(void) { return n_events; }
const char *fake_event(int i, char *kind, int *dev, unsigned *grid, size_t *smem, size_t *bytes) {
    *kind = events[i].kind, *dev = events[i].device, *grid = events[i].grid, *smem = events[i].smem, *bytes = events[i].bytes;
    return events[i].func >= 0 ? funcs[events[i].func].name : "";
}
/* copies to the host of `bytes` bytes arrive with `value` at `offset` */
void fake_patch(uint64_t bytes, uint64_t offset, uint64_t value) { patch_bytes = bytes, patch_offset = offset, patch_value = value; }

/* memory */
static int take(void **p, size_t n, int dev) {
    void *q = mmap(NULL, n ? n : 1, PROT_READ | PROT_WRITE, MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
    if (q == MAP_FAILED || n_blocks == BLOCKS) return fail(NO_MEMORY);
    blocks[n_blocks].p = q, blocks[n_blocks].n = n, blocks[n_blocks++].dev = dev;
    *p = q;
    return OK;
}
static int give(void *p) {
    for (int i = 0; i < n_blocks; ++i)
        if (blocks[i].p == p) {
            if (blocks[i].dev >= 0) used[blocks[i].dev] -= blocks[i].n;
            munmap(p, blocks[i].n ? blocks[i].n : 1);
            blocks[i] = blocks[--n_blocks];
            return OK;
        }
    return p ? fail(INVALID) : OK;
}
int cudaMalloc(void **p, size_t n) {
    if (used[device] + n > budget[device]) return fail(NO_MEMORY);
    const int e = take(p, n, device);
    if (!e) used[device] += n, note('M', -1, 0, 0, n);
    return e;
}
int cudaFree(void *p) { return give(p); }
int cudaHostAlloc(void **p, size_t n, unsigned flags) { return (void)flags, take(p, n, -1); }
int cudaMallocHost(void **p, size_t n) { return take(p, n, -1); }
int cudaFreeHost(void *p) { return give(p); }
int cudaMemGetInfo(size_t *f, size_t *t) { return *f = budget[device] - used[device], *t = budget[device], OK; }
int cudaMemcpy(void *d, const void *s, size_t n, int kind) {
    memcpy(d, s, n);
    if (kind == 2 && patch_bytes && n == patch_bytes) memcpy((char *)d + patch_offset, &patch_value, 8);
    return OK;
}
int cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st) { return (void)st, cudaMemcpy(d, s, n, kind); }
int cudaMemsetAsync(void *d, int v, size_t n, void *st) {
    (void)st;
    if (n <= 1 << 26) memset(d, v, n); /* (memory starts out clear) */
    return OK;
}
struct attrs { int type, device; void *dev_p, *host_p; long reserved[8]; };
int cudaPointerGetAttributes(struct attrs *a, const void *p) { return a->type = 0, a->dev_p = NULL, (void)p, OK; }
static char symbol[64 << 20];
int cudaGetSymbolAddress(void **p, const void *s) { return (void)s, *p = symbol, OK; }

/* devices, streams, events, graphs */
int cudaGetDevice(int *d) { return *d = device, OK; }
int cudaSetDevice(int d) { return d < DEVICES ? (device = d, OK) : fail(101); }
int cudaDeviceGetAttribute(int *v, int a, int d) { return (void)a, (void)d, *v = 152, OK; }
int cudaDeviceGetLimit(size_t *v, int l) { return (void)l, *v = 64, OK; }
int cudaDeviceSetLimit(int l, size_t v) { return (void)l, (void)v, OK; }
int cudaGetLastError(void) { const int e = last_error; return last_error = OK, e; }
static char handle;
#define SAME(name, ...) int name(__VA_ARGS__) { return OK; }
int cudaEventCreate(void **e) { return *e = &handle, OK; }
int cudaEventCreateWithFlags(void **e, unsigned f) { return (void)f, *e = &handle, OK; }
int cudaStreamCreateWithFlags(void **s, unsigned f) { return (void)f, *s = &handle, OK; }
int cudaEventElapsedTime(float *ms, void *a, void *b) { return (void)a, (void)b, *ms = 1, OK; }
int cudaStreamEndCapture(void *s, void **g) { return (void)s, *g = &handle, OK; }
int cudaGraphInstantiate(void **x, void *g, unsigned long long f) { return (void)g, (void)f, *x = &handle, OK; }
SAME(cudaEventDestroy, void *e) SAME(cudaEventQuery, void *e) SAME(cudaEventRecord, void *e, void *s)
SAME(cudaEventRecordWithFlags, void *e, void *s, unsigned f) SAME(cudaEventSynchronize, void *e)
SAME(cudaStreamSynchronize, void *s) SAME(cudaStreamDestroy, void *s) SAME(cudaStreamWaitEvent, void *s, void *e, unsigned f)
SAME(cudaStreamBeginCapture, void *s, int m) SAME(cudaGraphDestroy, void *g) SAME(cudaGraphExecDestroy, void *g)
SAME(cudaGraphLaunch, void *g, void *s)

/* kernels */
static int used_func(const void *f) {
    const int i = find(f);
    if (i < 0) return fail(98);
    note('F', i, 0, 0, 0);
    return OK;
}
int cudaFuncGetAttributes(void *a, const void *f) { return (void)a, used_func(f); }
int cudaFuncSetAttribute(const void *f, int attr, int v) {
    const int e = used_func(f);
    if (!e && attr == 8) funcs[find(f)].smem[device] = v;
    return e;
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int threads, size_t smem, unsigned flags) {
    (void)flags;
    const int by_threads = 2048 / threads, by_smem = smem ? (int)((228 << 10) / (smem + 1024)) : by_threads;
    *n = by_threads < by_smem ? by_threads : by_smem;
    return used_func(f);
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int threads, size_t smem) {
    return cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(n, f, threads, smem, 0);
}
static struct { dim3_t grid, block; size_t smem; void *stream; } config;
unsigned __cudaPushCallConfiguration(dim3_t g, dim3_t b, size_t smem, void *s) {
    return config.grid = g, config.block = b, config.smem = smem, config.stream = s, 0;
}
int __cudaPopCallConfiguration(dim3_t *g, dim3_t *b, size_t *smem, void *s) {
    return *g = config.grid, *b = config.block, *smem = config.smem, *(void **)s = config.stream, OK;
}
int __cudaGetKernel(void **k, const void *f) { return *k = (void *)f, OK; }
int __cudaLaunchKernel(void *k, dim3_t g, dim3_t b, void **args, size_t smem, void *s) {
    const int i = find(k);
    (void)args, (void)s;
    if (i < 0) return fail(98);
    if (!g.x || !b.x || b.x > 1024 || (smem > 48 << 10 && smem > (size_t)funcs[i].smem[device])) return fail(INVALID);
    note('L', i, g.x, smem, 0);
    return OK;
}
int cudaLaunchKernel(const void *f, dim3_t g, dim3_t b, void **args, size_t smem, void *s) {
    return __cudaLaunchKernel((void *)f, g, b, args, smem, s);
}
void **__cudaRegisterFatBinary(void *f) { static void *h; return (void)f, &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
char __cudaInitModule(void **h) { return (void)h, 1; }
void __cudaRegisterVar(void **h, char *v, char *a, const char *n, int e, size_t s, int c, int g) {
    (void)h, (void)v, (void)a, (void)n, (void)e, (void)s, (void)c, (void)g;
}
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int lim, void *t, void *b, void *bd, void *gd, int *w) {
    (void)h, (void)dev, (void)lim, (void)t, (void)b, (void)bd, (void)gd, (void)w;
    if (n_funcs < FUNCS) funcs[n_funcs].host = host, funcs[n_funcs++].name = name;
}
