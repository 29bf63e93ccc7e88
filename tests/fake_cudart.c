/* A stand-in for the CUDA runtime for host tests: device memory is host memory, copies are memcpy, and a kernel
 * launch only adds a line "device kernel grid.x block.x" to a log. It takes the place of libcudart when it is loaded
 * first under the same soname (tests/fake_cuda.py). */
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

typedef struct { unsigned x, y, z; } dim3_;

static int g_device = 0;
static char* g_log = NULL;
static size_t g_len = 0, g_cap = 0;
static struct { const void* fun; const char* name; } g_kernel[4096];
static int g_kernels = 0;
static dim3_ g_grid, g_block;

const char* fake_log(void) { return g_log ? g_log : ""; }
void fake_clear(void) { g_len = 0; if (g_log) g_log[0] = 0; }
void fake_set_device(int d) { g_device = d; }

static int launch(const void* fun, dim3_ grid, dim3_ block) {
    const char* name = "?";
    for (int i = 0; i < g_kernels; ++i)
        if (g_kernel[i].fun == fun) name = g_kernel[i].name;
    const size_t need = g_len + strlen(name) + 64;
    if (need > g_cap) {
        g_cap = 2 * need;
        g_log = realloc(g_log, g_cap);
    }
    g_len += (size_t)sprintf(g_log + g_len, "%d %s %u %u\n", g_device, name, grid.x, block.x);
    return 0;
}

/* registration and launches */
void** __cudaRegisterFatBinary(void* b) { static void* h; (void)b; return &h; }
void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
void __cudaUnregisterFatBinary(void** h) { (void)h; }
void __cudaRegisterVar(void) {}
void __cudaRegisterFunction(void** h, const char* fun, char* dfun, const char* name) {
    (void)h; (void)dfun;
    if (g_kernels < 4096) {
        g_kernel[g_kernels].fun = fun;
        g_kernel[g_kernels++].name = name;
    }
}
unsigned __cudaPushCallConfiguration(dim3_ grid, dim3_ block, size_t smem, void* stream) {
    (void)smem; (void)stream;
    g_grid = grid;
    g_block = block;
    return 0;
}
int __cudaPopCallConfiguration(dim3_* grid, dim3_* block, size_t* smem, void* stream) {
    *grid = g_grid;
    *block = g_block;
    *smem = 0;
    *(void**)stream = NULL;
    return 0;
}
int __cudaGetKernel(const void** k, const void* fun) { *k = fun; return 0; }
int __cudaLaunchKernel(const void* f, dim3_ g, dim3_ b, void** a, size_t s, void* st) {
    (void)a; (void)s; (void)st;
    return launch(f, g, b);
}
int cudaLaunchKernel(const void* f, dim3_ g, dim3_ b, void** a, size_t s, void* st) {
    (void)a; (void)s; (void)st;
    return launch(f, g, b);
}
int cudaLaunchKernelExC(const dim3_* cfg, const void* f, void** a) { (void)a; return launch(f, cfg[0], cfg[1]); }

/* device */
int cudaSetDevice(int d) { g_device = d; return 0; }
int cudaGetDevice(int* d) { *d = g_device; return 0; }
int cudaDeviceGetAttribute(int* v, int a, int d) { (void)d; *v = a == 16 ? 152 : 1; return 0; } /* 16: SM count */
int cudaFuncGetAttributes(void* a, const void* f) { (void)f; memset(a, 0, 64); return 0; }
int cudaFuncSetAttribute(void) { return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n) { *n = 2; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n) { *n = 2; return 0; }
int cudaOccupancyMaxActiveClusters(int* n) { *n = 152; return 0; }
int cudaGetLastError(void) { return 0; }
int cudaGetDriverEntryPointByVersion(void) { return 1; }
int cudaGetSymbolAddress(void) { return 1; }

/* memory: every pointer counts as device memory */
int cudaMalloc(void** p, size_t n) { *p = calloc(1, n ? n : 1); return *p ? 0 : 2; }
int cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
int cudaFree(void* p) { free(p); return 0; }
int cudaFreeHost(void* p) { free(p); return 0; }
int cudaMemcpy(void* d, const void* s, size_t n) { memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void* d, const void* s, size_t n) { memcpy(d, s, n); return 0; }
int cudaMemsetAsync(void* d, int v, size_t n) { memset(d, v, n); return 0; }
int cudaPointerGetAttributes(int* a) { *a = 2; return 0; } /* type: device */

/* streams, events, graphs */
static int handle(void** p) { static long n = 0; *p = (void*)(++n); return 0; }
int cudaStreamCreateWithFlags(void** p) { return handle(p); }
int cudaEventCreate(void** p) { return handle(p); }
int cudaEventCreateWithFlags(void** p) { return handle(p); }
int cudaStreamEndCapture(void* st, void** p) { (void)st; return handle(p); }
int cudaGraphInstantiate(void** p) { return handle(p); }
int cudaEventElapsedTime(float* ms) { *ms = 1.0f; return 0; }
int cudaStreamDestroy(void) { return 0; }
int cudaStreamSynchronize(void) { return 0; }
int cudaStreamWaitEvent(void) { return 0; }
int cudaStreamBeginCapture(void) { return 0; }
int cudaEventDestroy(void) { return 0; }
int cudaEventRecord(void) { return 0; }
int cudaEventRecordWithFlags(void) { return 0; }
int cudaEventSynchronize(void) { return 0; }
int cudaGraphDestroy(void) { return 0; }
int cudaGraphExecDestroy(void) { return 0; }
int cudaGraphLaunch(void) { return 0; }
