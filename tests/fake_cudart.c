/* CUDA runtime stand-in for tests of the library's host code without a GPU: preloaded before libcudart, it backs device
 * memory by host memory, runs no kernel and writes every allocation, fill, copy and launch to the file FAKE_CUDART_LOG:
 *   malloc PTR BYTES | memset PTR BYTES | memcpy DST SRC BYTES | launch NAME GRID BLOCK SMEM ARG ARG ...
 * A launch's arguments are the first 8 bytes of each of the leading parameters that FAKE_CUDART_ARGS asks for, as
 * "substring of the kernel's name:count" entries with commas between them. */
#include <cuda_runtime_api.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#define API __attribute__((visibility("default")))
#define MAX_KERNELS 4096

static struct { const void* fun; const char* name; } kernels[MAX_KERNELS];
static int n_kernels;
static FILE* out;

static FILE* log_file(void)
{
    if (!out) {
        const char* p = getenv("FAKE_CUDART_LOG");
        out = p ? fopen(p, "w") : stderr;
        setvbuf(out, NULL, _IOLBF, 0);
    }
    return out;
}

static void log_launch(const void* fun, dim3 g, dim3 b, size_t smem, void** args)
{
    const char* name = "?";
    for (int i = 0; i < n_kernels; ++i)
        if (kernels[i].fun == fun) name = kernels[i].name;
    fprintf(log_file(), "launch %s %u,%u,%u %u,%u,%u %zu", name, g.x, g.y, g.z, b.x, b.y, b.z, smem);
    const char* want = getenv("FAKE_CUDART_ARGS");
    char spec[512];
    snprintf(spec, sizeof spec, "%s", want ? want : "");
    for (char* s = strtok(spec, ","); s; s = strtok(NULL, ",")) {
        char* colon = strchr(s, ':');
        if (!colon) continue;
        *colon = 0;
        if (!strstr(name, s)) continue;
        for (int i = 0; i < atoi(colon + 1); ++i) {
            unsigned long long v = 0;
            memcpy(&v, args[i], 8);
            fprintf(log_file(), " %llu", v);
        }
        break;
    }
    fputc('\n', log_file());
}

API void** __cudaRegisterFatBinary(void* f) { static void* h; (void)f; return &h; }
API void __cudaRegisterFatBinaryEnd(void** h) { (void)h; }
API void __cudaUnregisterFatBinary(void** h) { (void)h; }
API void __cudaRegisterVar(void** h, char* v, char* d, const char* n, int e, size_t s, int c, int g)
{
    (void)h; (void)v; (void)d; (void)n; (void)e; (void)s; (void)c; (void)g;
}
API void __cudaRegisterFunction(void** h, const char* fun, char* dev, const char* name, int limit, void* tid, void* bid,
                                void* bd, void* gd, int* ws)
{
    (void)h; (void)dev; (void)limit; (void)tid; (void)bid; (void)bd; (void)gd; (void)ws;
    if (n_kernels < MAX_KERNELS) {
        kernels[n_kernels].fun = fun;
        kernels[n_kernels++].name = name;
    }
}

static dim3 cfg_g, cfg_b;
static size_t cfg_smem;
static cudaStream_t cfg_s;
API unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* s)
{
    cfg_g = g, cfg_b = b, cfg_smem = smem, cfg_s = s;
    return 0;
}
API cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s)
{
    *g = cfg_g, *b = cfg_b, *smem = cfg_smem, *(cudaStream_t*)s = cfg_s;
    return cudaSuccess;
}
API cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fun) { *k = (cudaKernel_t)fun; return cudaSuccess; }
API cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** args, size_t smem, cudaStream_t s)
{
    (void)s;
    log_launch((const void*)k, g, b, smem, args);
    return cudaSuccess;
}
API cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fun, void** args)
{
    log_launch(fun, c->gridDim, c->blockDim, c->dynamicSmemBytes, args);
    return cudaSuccess;
}

API cudaError_t cudaMalloc(void** p, size_t n)
{
    *p = aligned_alloc(512, (n + 511) / 512 * 512 + 512);
    if (!*p) return cudaErrorMemoryAllocation;
    memset(*p, 0, n);
    fprintf(log_file(), "malloc %llu %zu\n", (unsigned long long)*p, n);
    return cudaSuccess;
}
API cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
API cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s)
{
    (void)s;
    memset(p, v, n);
    fprintf(log_file(), "memset %llu %zu\n", (unsigned long long)p, n);
    return cudaSuccess;
}
API cudaError_t cudaMemset(void* p, int v, size_t n) { return cudaMemsetAsync(p, v, n, 0); }
API cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind k, cudaStream_t st)
{
    (void)k; (void)st;
    memmove(d, s, n);
    fprintf(log_file(), "memcpy %llu %llu %zu\n", (unsigned long long)d, (unsigned long long)s, n);
    return cudaSuccess;
}
API cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind k) { return cudaMemcpyAsync(d, s, n, k, 0); }

API cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
API cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
API cudaError_t cudaSetDevice(int d) { (void)d; return cudaSuccess; }
API cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d)
{
    (void)d;
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
API cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v)
{
    (void)f; (void)a; (void)v;
    return cudaSuccess;
}
API cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int b, size_t s, unsigned fl)
{
    (void)f; (void)b; (void)s; (void)fl;
    *n = 2;
    return cudaSuccess;
}
API cudaError_t cudaGetLastError(void) { return cudaSuccess; }
API const char* cudaGetErrorString(cudaError_t e) { (void)e; return "stand-in"; }
API cudaError_t cudaGetSymbolAddress(void** p, const void* s)
{
    static char buf[1 << 23];
    (void)s;
    *p = buf;
    return cudaSuccess;
}
API cudaError_t cudaStreamSynchronize(cudaStream_t s) { (void)s; return cudaSuccess; }
API cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus* c)
{
    (void)s;
    *c = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
API cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned f) { (void)f; *s = (cudaStream_t)8; return cudaSuccess; }
API cudaError_t cudaStreamDestroy(cudaStream_t s) { (void)s; return cudaSuccess; }
API cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned f) { (void)s; (void)e; (void)f; return cudaSuccess; }
API cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = (cudaEvent_t)8; return cudaSuccess; }
API cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned f) { (void)f; *e = (cudaEvent_t)8; return cudaSuccess; }
API cudaError_t cudaEventDestroy(cudaEvent_t e) { (void)e; return cudaSuccess; }
API cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { (void)e; (void)s; return cudaSuccess; }
API cudaError_t cudaEventSynchronize(cudaEvent_t e) { (void)e; return cudaSuccess; }
