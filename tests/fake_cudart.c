/* A stand-in for the CUDA runtime's host calls, preloaded over libcudart by
 * the CPU tests of the launchers: `wq4_fake_device` devices that accept every
 * launch whose dynamic shared memory is within what was set for that kernel
 * on the current device.  Nothing runs; device pointers are never read. */
#include <cuda.h>
#include <cuda_runtime_api.h>

enum { kDevices = 4, kKernels = 256 };

static int g_device;
static const void* g_kernel[kKernels];
static int g_limit[kKernels][kDevices];
static unsigned g_word[kDevices];
static int g_launches;
static int g_last = -1;
static size_t g_last_shape;

static int kernel_index(const void* f)
{
    int i = 0;
    while (i < kKernels - 1 && g_kernel[i] && g_kernel[i] != f) ++i;
    g_kernel[i] = f;
    return i;
}

static cudaError_t launch(const void* f, dim3 grid, size_t smem)
{
    const int i = kernel_index(f);
    if (grid.x < 1 || grid.x > 0x7FFFFFFFu || grid.y < 1 || grid.y > 65535u) return cudaErrorInvalidConfiguration;
    if (smem > 48 * 1024 && smem > (size_t)g_limit[i][g_device]) return cudaErrorInvalidValue;
    ++g_launches;
    g_last = i;
    g_last_shape = (size_t)grid.x << 32 | smem;
    return cudaSuccess;
}

void fake_set_device(int d) { g_device = d; }
int fake_launches(void) { return g_launches; }
int fake_last_kernel(void) { return g_last; }
size_t fake_last_shape(void) { return g_last_shape; }   /* grid << 32 | shared memory */

cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }

cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d)
{
    (void)d;
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 1;
    return cudaSuccess;
}

cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v)
{
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_limit[kernel_index(f)][g_device] = v;
    return cudaSuccess;
}

cudaError_t cudaGetSymbolAddress(void** p, const void* symbol)
{
    (void)symbol;
    *p = &g_word[g_device];
    return cudaSuccess;
}

cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c)
{
    (void)f;
    *n = 152 / (int)c->attrs[0].val.clusterDim.x;
    return cudaSuccess;
}

cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int threads, size_t smem,
                                                                    unsigned flags)
{
    (void)f, (void)threads, (void)smem, (void)flags;
    *n = 2;
    return cudaSuccess;
}

static CUresult encode_tiled(CUtensorMap* m, CUtensorMapDataType t, cuuint32_t rank, void* base, const cuuint64_t* dims,
                             const cuuint64_t* strides, const cuuint32_t* box, const cuuint32_t* es,
                             CUtensorMapInterleave i, CUtensorMapSwizzle s, CUtensorMapL2promotion l,
                             CUtensorMapFloatOOBfill o)
{
    (void)m, (void)t, (void)dims, (void)es, (void)i, (void)s, (void)l, (void)o;
    if ((size_t)base % 16) return CUDA_ERROR_INVALID_VALUE;
    for (cuuint32_t r = 0; r < rank; ++r)
        if (box[r] < 1 || box[r] > 256 || (r > 0 && strides[r - 1] % 16)) return CUDA_ERROR_INVALID_VALUE;
    return CUDA_SUCCESS;
}

cudaError_t cudaGetDriverEntryPoint(const char* name, void** p, unsigned long long flags,
                                    enum cudaDriverEntryPointQueryResult* q)
{
    (void)name, (void)flags;
    *p = (void*)encode_tiled;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }

cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t s)
{
    (void)block, (void)args, (void)s;
    return launch((const void*)k, grid, smem);
}

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args)
{
    (void)args;
    return launch(f, c->gridDim, c->dynamicSmemBytes);
}
