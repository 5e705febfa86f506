// A CUDA runtime without a GPU, preloaded before libcudart: "device" memory is host
// memory, launches are counted instead of run, and calls can be made to fail. The
// last error is kept as the runtime keeps it: set by a failing call, returned and
// cleared by cudaGetLastError().
#include <stdlib.h>
#include <string.h>

#include <cuda_runtime_api.h>

static int n_launches;
static cudaError_t last_error;
// calls of the kind still to be refused: 0 launches, 1 cudaFuncSetAttribute, 2 cudaFuncGetAttributes
static int refuse[3];

static cudaError_t done(cudaError_t e) {
    if (e != cudaSuccess) last_error = e;
    return e;
}
static int refused(int kind) { return refuse[kind] > 0 && refuse[kind]-- > 0; }

// ---- for the tests ----
void fake_refuse(int kind, int times) { refuse[kind] = times; }
int fake_launches(void) { return n_launches; }
int fake_pending_error(void) { return (int)last_error; }

// ---- the runtime's calls ----
cudaError_t cudaGetLastError(void) {
    const cudaError_t e = last_error;
    last_error = cudaSuccess;
    return e;
}
cudaError_t cudaGetDevice(int *dev) { *dev = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int dev) { return done(dev == 0 ? cudaSuccess : cudaErrorInvalidDevice); }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr attr, int dev) {
    (void)dev;
    *v = attr == cudaDevAttrMultiProcessorCount ? 152 : 227 * 1024;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n) {
    *p = aligned_alloc(256, (n + 255) / 256 * 256);
    return done(*p ? cudaSuccess : cudaErrorMemoryAllocation);
}
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind k) {
    (void)k;
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t st) {
    (void)st;
    return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t st) {
    (void)st;
    memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t st) { (void)st; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **p, const void *symbol) {
    static char memory[1 << 18];
    (void)symbol;
    *p = memory;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v) {
    (void)f; (void)a; (void)v;
    return done(refused(1) ? cudaErrorInvalidValue : cudaSuccess);
}
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes *a, const void *f) {
    (void)f;
    memset(a, 0, sizeof *a);
    a->numRegs = 96;
    return done(refused(2) ? cudaErrorInvalidValue : cudaSuccess);
}
static cudaError_t launch(void) {
    if (refused(0)) return done(cudaErrorInvalidConfiguration);
    n_launches++;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args) {
    (void)c; (void)f; (void)args;
    return launch();
}

// ---- what <<<>>> and the registration of a library's kernels turn into ----
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t st) {
    (void)k; (void)grid; (void)block; (void)args; (void)smem; (void)st;
    return launch();
}
static dim3 pushed_grid, pushed_block;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void *st) {
    (void)smem; (void)st;
    pushed_grid = grid;
    pushed_block = block;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *st) {
    *grid = pushed_grid;
    *block = pushed_block;
    *smem = 0;
    *(void **)st = 0;
    return cudaSuccess;
}
void **__cudaRegisterFatBinary(void *image) { static void *handle; (void)image; return &handle; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterFunction(void **h, const char *host, char *dev, const char *name, int limit, void *tid, void *bid,
                            void *bdim, void *gdim, int *wsize) {
    (void)h; (void)host; (void)dev; (void)name; (void)limit; (void)tid; (void)bid; (void)bdim; (void)gdim; (void)wsize;
}
void __cudaRegisterVar(void **h, char *host, char *dev, const char *name, int ext, size_t size, int constant, int global) {
    (void)h; (void)host; (void)dev; (void)name; (void)ext; (void)size; (void)constant; (void)global;
}
