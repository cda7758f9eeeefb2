/* The part of the CUDA runtime that the library's objects import, for host
   tests of its launch logic without a GPU: device memory is host memory,
   kernels do not run, and every launch is handed to the test, which may fail
   it. Declarations follow cuda_runtime_api.h and crt/host_runtime.h. */
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3_t;
typedef struct { dim3_t grid, block; size_t smem; void *stream; void *attrs; unsigned num_attrs; } config_t;

/* launch(kernel name, parameter pointers) and memset(pointer, value, bytes) return a cudaError_t */
typedef int (*launch_fn)(const char *name, void **args);
typedef int (*memset_fn)(void *p, int value, size_t n);
static launch_fn on_launch;
static memset_fn on_memset;
static int capturing;
void fake_hooks(launch_fn l, memset_fn m) { on_launch = l; on_memset = m; }
void fake_capturing(int yes) { capturing = yes; }

/* host stub -> kernel name */
static struct { const void *fn; const char *name; } kernels[1024];
static int n_kernels;

void **__cudaRegisterFatBinary(void *bin) { static void *handle; (void)bin; return &handle; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int limit, void *tid, void *bid,
                            void *bdim, void *gdim, int *wsize) {
    (void)h; (void)dev; (void)limit; (void)tid; (void)bid; (void)bdim; (void)gdim; (void)wsize;
    if (n_kernels < 1024) {
        kernels[n_kernels].fn = host;
        kernels[n_kernels++].name = name;
    }
}
void __cudaRegisterVar(void **h, char *var, char *addr, const char *name, int ext, size_t size, int constant, int global) {
    (void)h; (void)var; (void)addr; (void)name; (void)ext; (void)size; (void)constant; (void)global;
}

static int launch(const void *fn, void **args) {
    const char *name = "?";
    for (int k = 0; k < n_kernels; ++k)
        if (kernels[k].fn == fn) name = kernels[k].name;
    return on_launch ? on_launch(name, args) : 0;
}
int cudaLaunchKernelExC(const config_t *c, const void *fn, void **args) { (void)c; return launch(fn, args); }
int __cudaGetKernel(void **kernel, const void *fn) { *kernel = (void *)fn; return 0; }
int __cudaLaunchKernel(void *kernel, dim3_t g, dim3_t b, void **args, size_t smem, void *stream) {
    (void)g; (void)b; (void)smem; (void)stream;
    return launch(kernel, args);
}
static struct { dim3_t g, b; size_t smem; void *stream; } pushed;
unsigned __cudaPushCallConfiguration(dim3_t g, dim3_t b, size_t smem, void *stream) {
    pushed.g = g; pushed.b = b; pushed.smem = smem; pushed.stream = stream;
    return 0;
}
int __cudaPopCallConfiguration(dim3_t *g, dim3_t *b, size_t *smem, void *stream) {
    *g = pushed.g; *b = pushed.b; *smem = pushed.smem; *(void **)stream = pushed.stream;
    return 0;
}

int cudaMalloc(void **p, size_t n) { *p = calloc(n ? n : 1, 1); return *p ? 0 : 2; }
int cudaFree(void *p) { free(p); return 0; }
int cudaMemset(void *p, int v, size_t n) { memset(p, v, n); return 0; }
int cudaMemsetAsync(void *p, int v, size_t n, void *s) {
    (void)s;
    const int e = on_memset ? on_memset(p, v, n) : 0;
    if (e == 0) memset(p, v, n);
    return e;
}
int cudaMemcpy(void *d, const void *s, size_t n, int kind) { (void)kind; memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st) { (void)st; return cudaMemcpy(d, s, n, kind); }
int cudaGetSymbolAddress(void **p, const void *sym) { (void)sym; *p = 0; return 1; }
int cudaGetLastError(void) { return 0; }
const char *cudaGetErrorString(int e) { return e == 2 ? "out of memory" : e ? "error" : "no error"; }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaSetDevice(int d) { (void)d; return 0; }
int cudaDeviceSynchronize(void) { return 0; }
int cudaDeviceGetAttribute(int *v, int attr, int dev) { (void)attr; (void)dev; *v = 152; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int t, size_t s) {
    (void)f; (void)t; (void)s;
    *n = 4;
    return 0;
}
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int t, size_t s, unsigned fl) {
    (void)fl;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, t, s);
}
int cudaEventRecord(void *e, void *s) { (void)e; (void)s; return 0; }
int cudaStreamSynchronize(void *s) { (void)s; return 0; }
int cudaStreamIsCapturing(void *s, int *status) { (void)s; *status = capturing; return 0; }
