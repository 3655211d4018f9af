/* A CUDA runtime with one device and no GPU behind it, preloaded in front of the real one by
 * tests/test_launch_host.py: the host code of the library runs as with a GPU, no kernel is executed, and
 * launches and attribute calls are written to a log, one line each.
 *   attr <kernel> <bytes>                           cudaFuncSetAttribute
 *   launch <kernel> <grid.x> <threads> <bytes> <cluster> [<claims>]
 * (claims, of the block kernels: 1 where the launch is given the counter that tasks are claimed from)
 */
#include <driver_types.h>
#include <stddef.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

enum { kKernels = 2048, kLog = 1 << 22 };
static const void *fun_of[kKernels];
static const char *name_of[kKernels];
static int kernels;
static char log_text[kLog];
static size_t log_used;

const char *fake_log(void)
{
    log_text[log_used] = 0;
    log_used = 0;
    return log_text;
}

static const char *kernel_name(const void *f)
{
    for (int i = 0; i < kernels; ++i) if (fun_of[i] == f) return name_of[i];
    return "?";
}

#define LOG(...) do { if (log_used < kLog - 4096) log_used += (size_t)snprintf(log_text + log_used, 4096, __VA_ARGS__); } while (0)

void **__cudaRegisterFatBinary(void *p) { static void *h; (void)p; return &h; }
void __cudaRegisterFatBinaryEnd(void **h) { (void)h; }
void __cudaUnregisterFatBinary(void **h) { (void)h; }
void __cudaRegisterVar(void **h, char *a, char *b, const char *c, int d, size_t e, int f, int g)
{ (void)h; (void)a; (void)b; (void)c; (void)d; (void)e; (void)f; (void)g; }
void __cudaRegisterFunction(void **h, const char *fun, char *dev_fun, const char *name, int limit, void *a, void *b, void *c, void *d, int *e)
{
    (void)h; (void)dev_fun; (void)limit; (void)a; (void)b; (void)c; (void)d; (void)e;
    if (kernels < kKernels) { fun_of[kernels] = fun; name_of[kernels++] = name; }
}
unsigned __cudaPushCallConfiguration(struct dim3 g, struct dim3 b, size_t s, void *st) { (void)g; (void)b; (void)s; (void)st; return 0; }
int __cudaPopCallConfiguration(struct dim3 *g, struct dim3 *b, size_t *s, void *st) { (void)g; (void)b; (void)s; (void)st; return 1; }

int cudaGetDeviceCount(int *n) { *n = 1; return 0; }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaGetLastError(void) { return 0; }
const char *cudaGetErrorString(int e) { (void)e; return "fake"; }

/* What a context keeps on the device: the last allocation, which tests look into. */
static unsigned char *device_block;
static size_t device_block_bytes;
void *fake_device_block(size_t *bytes) { *bytes = device_block_bytes; return device_block; }
int cudaMalloc(void **p, size_t n)
{
    *p = aligned_alloc(256, (n + 255) & ~(size_t)255);
    device_block = *p;
    device_block_bytes = n;
    return *p ? 0 : 2;
}
int cudaFree(void *p) { free(p); return 0; }
int cudaMemcpy(void *d, const void *s, size_t n, int kind) { (void)kind; memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int kind, void *st) { (void)kind; (void)st; memcpy(d, s, n); return 0; }
int cudaMemsetAsync(void *p, int v, size_t n, void *st) { (void)st; memset(p, v, n); return 0; }
int cudaDeviceSynchronize(void) { return 0; }
int cudaStreamSynchronize(void *st) { (void)st; return 0; }
int cudaGetSymbolAddress(void **p, const void *s) { *p = (void *)s; return 0; }

/* the figures of a B200 */
int cudaDeviceGetAttribute(int *v, int attr, int dev)
{
    (void)dev;
    *v = attr == cudaDevAttrMultiProcessorCount ? 148
         : attr == cudaDevAttrMaxSharedMemoryPerMultiprocessor ? 233472
         : attr == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448
         : attr == cudaDevAttrReservedSharedMemoryPerBlock ? 1024 : 0;
    return 0;
}

int cudaFuncSetAttribute(const void *f, int attr, int value)
{
    if (attr == cudaFuncAttributeMaxDynamicSharedMemorySize) LOG("attr %s %d\n", kernel_name(f), value);
    return 0;
}

/* What a B200 answers for kernels of 128 registers per thread: four CTAs of 128 threads or two of 256 per SM,
 * less where shared memory is short; clusters of eight do not fill the SMs. */
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int threads, size_t smem)
{
    (void)f;
    const int by_smem = (int)(233472 / (smem + 1024)), by_regs = 512 / threads;
    *n = by_smem < by_regs ? by_smem : by_regs;
    return 0;
}

int cudaOccupancyMaxActiveClusters(int *n, const void *f, const cudaLaunchConfig_t *c)
{
    static const int of_eight[5] = {0, 15, 33, 48, 71};
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, (int)c->blockDim.x, c->dynamicSmemBytes);
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension)
            *n = c->attrs[i].val.clusterDim.x == 8 ? of_eight[*n] : 148 * *n / (int)c->attrs[i].val.clusterDim.x;
    return 0;
}

int cudaLaunchKernel(const void *f, struct dim3 g, struct dim3 b, void **args, size_t smem, void *st)
{
    (void)args; (void)st;
    LOG("launch %s %u %u %zu 1\n", kernel_name(f), g.x, b.x, smem);
    return 0;
}

/* BlockParams (the second argument): the context's device block, and two of its counters side by side, the one that
 * tasks are claimed from, or null, and that of the CTAs that have ended. */
static int block_claims(void **args)
{
    const uintptr_t *word = args[1], dev = word[3];
    for (int i = 4; i < 16; ++i) if (word[i] == dev + 256) return word[i - 1] == dev + 128;
    return -1;
}

int cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args)
{
    unsigned cluster = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i) if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.x;
    LOG("launch %s %u %u %zu %u", kernel_name(f), c->gridDim.x, c->blockDim.x, c->dynamicSmemBytes, cluster);
    if (strstr(kernel_name(f), "block_kernel") != NULL) LOG(" %d", block_claims(args));
    LOG("\n");
    return 0;
}

static int encode(void *map) { memset(map, 0, 128); return 0; }
int cudaGetDriverEntryPoint(const char *s, void **p, unsigned long long flags, int *q)
{
    (void)s; (void)flags;
    *p = (void *)(uintptr_t)encode;
    *q = 0;
    return 0;
}
