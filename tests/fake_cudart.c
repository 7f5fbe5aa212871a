/* The CUDA runtime calls that libdd.so makes while it plans, answered on the
 * host as a GB300 would answer them, for tests of plan-time decisions on a
 * machine without a GPU (preloaded before the real runtime, which still
 * registers the kernels). Nothing runs: "device" memory is host memory that no
 * one reads, launches are only recorded. */
#include <stdlib.h>
#include <string.h>

typedef int err_t;
typedef struct { unsigned x, y, z; } dim3_t;
/* one recorded launch: shape and the first bytes of the first argument */
typedef struct {
    dim3_t grid, block;
    size_t smem;
    unsigned char arg0[256];
} launch_t;

static launch_t launches[64], last;
static int n_launches;

int fake_launch_count(void) { return n_launches; }
const launch_t *fake_launch(int i) { return &launches[i]; }
void fake_launch_reset(void) { n_launches = 0; }

err_t cudaGetDevice(int *d) { *d = 0; return 0; }
err_t cudaDeviceGetAttribute(int *v, int attr, int d) {
    *v = attr == 16 ? 152 : (attr == 97 ? 227 * 1024 : 0); /* SMs, shared memory per block */
    return 0;
}
err_t cudaGetDeviceProperties(void *p, int d) {
    memset(p, 0, 256); /* the name comes first */
    strcpy(p, "fake");
    return 0;
}
err_t cudaStreamCreateWithFlags(void **s, unsigned f) { *s = NULL; return 0; }
err_t cudaStreamDestroy(void *s) { return 0; }
err_t cudaStreamSynchronize(void *s) { return 0; }
err_t cudaStreamWaitEvent(void *s, void *e, unsigned f) { return 0; }
err_t cudaStreamIsCapturing(void *s, int *st) { *st = 0; return 0; }
err_t cudaDeviceSynchronize(void) { return 0; }
err_t cudaEventCreate(void **e) { *e = (void *)1; return 0; }
err_t cudaEventCreateWithFlags(void **e, unsigned f) { *e = (void *)1; return 0; }
err_t cudaEventDestroy(void *e) { return 0; }
err_t cudaEventRecord(void *e, void *s) { return 0; }
err_t cudaEventSynchronize(void *e) { return 0; }
static err_t allocate(void **p) { return posix_memalign(p, 256, 256) ? 2 : 0; }
err_t cudaMalloc(void **p, size_t n) { return allocate(p); }
err_t cudaMallocAsync(void **p, size_t n, void *s) { return allocate(p); }
err_t cudaFree(void *p) { free(p); return 0; }
err_t cudaFreeAsync(void *p, void *s) { free(p); return 0; }
err_t cudaMemcpy(void *a, const void *b, size_t n, int k) { return 0; }
/* the last upload, for what it holds */
static unsigned char upload[8192];
static size_t upload_bytes;
const unsigned char *fake_upload(size_t *n) { *n = upload_bytes; return upload; }
err_t cudaMemcpyAsync(void *a, const void *b, size_t n, int k, void *s) {
    upload_bytes = n;
    memcpy(upload, b, n < sizeof upload ? n : sizeof upload);
    return 0;
}
err_t cudaMemset(void *a, int v, size_t n) { return 0; }
err_t cudaMemsetAsync(void *a, int v, size_t n, void *s) { return 0; }
err_t cudaFuncGetAttributes(void *a, const void *f) { memset(a, 0, 64); return 0; }
err_t cudaFuncSetAttribute(const void *f, int a, int v) { return 0; }
err_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int b, size_t s) {
    *n = 1;
    return 0;
}
err_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, size_t s,
                                                             unsigned fl) {
    *n = 1;
    return 0;
}
err_t cudaGraphCreate(void **g, unsigned f) { *g = (void *)1; return 0; }
err_t cudaGraphAddMemsetNode(void **n, void *g, void *const *d, size_t k, const void *p) {
    *n = (void *)1;
    return 0;
}
err_t cudaGraphAddKernelNode(void **n, void *g, void *const *d, size_t k, const void *p) {
    *n = (void *)1;
    return 0;
}
err_t cudaGraphInstantiate(void **e, void *g, unsigned long long f) { *e = (void *)1; return 0; }
err_t cudaGraphLaunch(void *e, void *s) { return 0; }
err_t cudaGraphExecDestroy(void *e) { return 0; }
err_t cudaGraphDestroy(void *g) { return 0; }
err_t cudaGetLastError(void) { return 0; }
err_t __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return 0; }
/* Milliseconds of the last forward launch, by its tile and launch order: 0.5 for
 * the favoured tile with time tiles fastest, 2 for it with DM tiles fastest, 1.5
 * and 1 for the others. (Offsets of FwdArgs: see fake_gpu.py.) */
static int favoured[3];
void fake_favour(int dt, int ts, int cch) {
    favoured[0] = dt;
    favoured[1] = ts;
    favoured[2] = cch;
}
err_t cudaEventElapsedTime(float *ms, void *a, void *b) {
    int shape[4], order;
    memcpy(shape, last.arg0 + 48, sizeof shape); /* Dt, Ts, C_pad, cch */
    memcpy(&order, last.arg0 + 108, sizeof order);
    const int hit = shape[0] == favoured[0] && shape[1] == favoured[1] && shape[3] == favoured[2];
    *ms = hit ? (order ? 0.5f : 2.0f) : (order ? 1.5f : 1.0f);
    return 0;
}
err_t __cudaLaunchKernel(void *f, dim3_t grid, dim3_t block, void **args, size_t smem, void *s) {
    if (smem) memcpy(last.arg0, args[0], sizeof last.arg0);
    if (n_launches < 64) {
        launch_t *l = &launches[n_launches++];
        l->grid = grid;
        l->block = block;
        l->smem = smem;
        memcpy(l->arg0, args[0], 8); /* every kernel's first argument has 8 bytes */
        if (smem) memcpy(l->arg0, args[0], sizeof l->arg0); /* forward kernels: FwdArgs */
    }
    return 0;
}
