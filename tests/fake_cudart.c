/* A stand-in for libcudart.so.13 on a machine without a GPU, for the host logic around the kernels: device memory is host
 * memory, streams, events and graphs are tokens, kernels are counted and not run (what they would write stays 0).  Calls are
 * counted by name, and fake_fail(name, skip) makes one call of that name fail after `skip` more that succeed. */
#include <stdlib.h>
#include <string.h>

typedef int err_t; /* cudaError_t */
enum { kNames = 64, kFailed = 1 };
static struct { const char *name; long calls; long fail_at; } table[kNames];
static int names;
static err_t last;

static int slot(const char *name) {
    for (int i = 0; i < names; ++i)
        if (!strcmp(table[i].name, name)) return i;
    table[names].name = strdup(name);
    table[names].fail_at = -1;
    return names++;
}
static err_t hit(const char *name) {
    const int i = slot(name);
    if (table[i].calls++ != table[i].fail_at) return 0;
    return last = kFailed;
}
long fake_calls(const char *name) { return table[slot(name)].calls; }
void fake_fail(const char *name, long skip) {
    const int i = slot(name);
    table[i].fail_at = table[i].calls + skip;
}

static err_t token(const char *name, void **out) {
    const err_t e = hit(name);
    if (!e) *out = calloc(1, 16);
    return e;
}
static err_t release(const char *name, void *p) {
    free(p);
    return hit(name);
}

err_t cudaGetLastError(void) {
    const err_t e = last;
    last = 0;
    return e;
}
const char *cudaGetErrorString(err_t e) { return e ? "fake failure" : "no error"; }
err_t cudaGetDevice(int *d) { return *d = 0; }
err_t cudaDeviceGetAttribute(int *v, int attr, int dev) { return *v = 152, 0; }
err_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int threads, size_t smem) { return *n = 2, 0; }
err_t cudaFuncSetAttribute(const void *f, int attr, int v) { return hit("cudaFuncSetAttribute"); }
err_t cudaGetSymbolAddress(void **p, const void *sym) { return token("cudaGetSymbolAddress", p); }

err_t cudaMalloc(void **p, size_t n) {
    const err_t e = hit("cudaMalloc");
    if (!e) *p = calloc(1, n);
    return e;
}
err_t cudaHostAlloc(void **p, size_t n, unsigned flags) { return *p = calloc(1, n), hit("cudaHostAlloc"); }
err_t cudaFree(void *p) { return release("cudaFree", p); }
err_t cudaFreeHost(void *p) { return release("cudaFreeHost", p); }
err_t cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st) { return memcpy(d, s, n), hit("cudaMemcpyAsync"); }
err_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, int kind, void *st) {
    return hit("cudaMemcpy2DAsync");
}
err_t cudaMemsetAsync(void *p, int v, size_t n, void *st) { return memset(p, v, n), hit("cudaMemsetAsync"); }

err_t cudaStreamCreateWithFlags(void **s, unsigned flags) { return token("cudaStreamCreateWithFlags", s); }
err_t cudaStreamDestroy(void *s) { return release("cudaStreamDestroy", s); }
err_t cudaStreamSynchronize(void *s) { return hit("cudaStreamSynchronize"); }
err_t cudaStreamWaitEvent(void *s, void *e, unsigned flags) { return hit("cudaStreamWaitEvent"); }
err_t cudaStreamIsCapturing(void *s, int *status) { return *status = 0, hit("cudaStreamIsCapturing"); }
err_t cudaStreamBeginCapture(void *s, int mode) { return hit("cudaStreamBeginCapture"); }
err_t cudaStreamEndCapture(void *s, void **graph) { return token("cudaStreamEndCapture", graph); }
err_t cudaGraphInstantiate(void **exec, void *graph, unsigned long long flags) { return token("cudaGraphInstantiate", exec); }
err_t cudaGraphLaunch(void *exec, void *s) { return hit("cudaGraphLaunch"); }
err_t cudaGraphDestroy(void *g) { return release("cudaGraphDestroy", g); }
err_t cudaGraphExecDestroy(void *g) { return release("cudaGraphExecDestroy", g); }
err_t cudaEventCreate(void **e) { return token("cudaEventCreate", e); }
err_t cudaEventCreateWithFlags(void **e, unsigned flags) { return token("cudaEventCreate", e); }
err_t cudaEventDestroy(void *e) { return release("cudaEventDestroy", e); }
err_t cudaEventRecord(void *e, void *s) { return hit("cudaEventRecord"); }
err_t cudaEventSynchronize(void *e) { return hit("cudaEventSynchronize"); }
err_t cudaEventElapsedTime(float *ms, void *a, void *b) { return *ms = 1.0f, hit("cudaEventElapsedTime"); }

/* launches: of triple-chevron calls and of cudaLaunchKernelEx */
err_t cudaLaunchKernelExC(const void *cfg, const void *f, void **args) { return hit("launch"); }
err_t __cudaLaunchKernel(void) { return hit("launch"); }
err_t __cudaGetKernel(void **k, const void *f) { return *k = (void *)f, 0; }
unsigned __cudaPushCallConfiguration(void) { return 0; }
err_t __cudaPopCallConfiguration(void *g, void *b, size_t *smem, void *st) { return 0; }
void **__cudaRegisterFatBinary(void *fat) {
    static void *handle[2];
    return handle;
}
void __cudaRegisterFatBinaryEnd(void **h) {}
void __cudaUnregisterFatBinary(void **h) {}
void __cudaRegisterFunction(void) {}
void __cudaRegisterVar(void) {}
