// A stand-in for the CUDA runtime, for host-side tests without a GPU: several devices, each kernel's dynamic shared
// memory opt-in kept per device as the real one keeps it, memory from the host heap, and launches that are checked
// and counted but run nothing.  Linked with the library's own objects in place of libcudart.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>

namespace {

constexpr int kDevices = 2, kOptin = 232448, kDefault = 48 * 1024;

int g_device = 0;
std::map<const void *, std::string> g_name;
std::map<std::pair<int, const void *>, int> g_limit;   // (device, kernel): dynamic shared memory allowed
long long g_launches = 0, g_refused = 0, g_lowered = 0, g_allocated = 0;
std::string g_first_refused, g_first_lowered;
cudaError_t g_last = cudaSuccess;

int limit(const void *f)
{
    const auto it = g_limit.find({g_device, f});
    return it == g_limit.end() ? kDefault : it->second;
}

cudaError_t launch(const void *f, size_t smem)
{
    ++g_launches;
    if (smem <= (size_t)limit(f))
        return cudaSuccess;
    if (!g_refused++)
        g_first_refused = g_name[f];
    return g_last = cudaErrorInvalidValue;
}

struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
} g_config;

}  // namespace

#define ALWAYS_OK(name, ...) cudaError_t name(__VA_ARGS__) { return cudaSuccess; }

extern "C" {

// what the tests read and set
void fake_set_device(int d) { g_device = d; }
long long fake_launches() { return g_launches; }
long long fake_refused() { return g_refused; }
long long fake_lowered() { return g_lowered; }
long long fake_allocated() { return g_allocated; }
const char *fake_first_refused() { return g_first_refused.c_str(); }
const char *fake_first_lowered() { return g_first_lowered.c_str(); }

// what compiled translation units call
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *)
{
    g_name[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st *stream)
{
    g_config = {grid, block, smem, stream};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream)
{
    *grid = g_config.grid;
    *block = g_config.block;
    *smem = g_config.smem;
    *(cudaStream_t *)stream = g_config.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *host)
{
    *k = (cudaKernel_t)host;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void **, size_t smem, cudaStream_t) { return launch((const void *)k, smem); }

// the runtime entry points the library uses
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **) { return launch(f, c->dynamicSmemBytes); }
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int value)
{
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize)
        return cudaSuccess;
    if (value < 0 || value > kOptin)
        return g_last = cudaErrorInvalidValue;
    if (value < limit(f) && !g_lowered++)
        g_first_lowered = g_name[f];
    g_limit[{g_device, f}] = value;
    return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *)
{
    std::memset(a, 0, sizeof(*a));
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d)
{
    *d = g_device;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int device)
{
    *v = a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? kOptin : a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return device >= 0 && device < kDevices ? cudaSuccess : cudaErrorInvalidDevice;
}
const char *cudaGetErrorString(cudaError_t) { return "refused by the stand-in runtime"; }
cudaError_t cudaGetLastError()
{
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaMallocHost(void **p, size_t n) { return (*p = std::calloc(n ? n : 1, 1)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMallocHost(p, n); }
cudaError_t cudaMalloc(void **p, size_t n)
{
    g_allocated += (long long)n;
    return cudaMallocHost(p, n);
}
cudaError_t cudaFree(void *p)
{
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t)
{
    *f = *t = (size_t)1 << 38;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind)
{
    std::memmove(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemset(void *d, int v, size_t n)
{
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaMemcpyToSymbol(const void *, const void *, size_t, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyFromSymbol(void *d, const void *, size_t n, size_t, cudaMemcpyKind) { return cudaMemset(d, 0, n); }
cudaError_t cudaGetSymbolAddress(void **p, const void *)
{
    static char symbol[1 << 16];
    *p = symbol;
    return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t)
{
    *ms = 0.0f;
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
ALWAYS_OK(cudaEventCreate, cudaEvent_t *)
ALWAYS_OK(cudaEventCreateWithFlags, cudaEvent_t *, unsigned)
ALWAYS_OK(cudaEventDestroy, cudaEvent_t)
ALWAYS_OK(cudaEventRecord, cudaEvent_t, cudaStream_t)
ALWAYS_OK(cudaEventSynchronize, cudaEvent_t)
ALWAYS_OK(cudaStreamCreateWithFlags, cudaStream_t *, unsigned)
ALWAYS_OK(cudaStreamDestroy, cudaStream_t)
ALWAYS_OK(cudaStreamSynchronize, cudaStream_t)
ALWAYS_OK(cudaStreamWaitEvent, cudaStream_t, cudaEvent_t, unsigned)
ALWAYS_OK(cudaStreamBeginCapture, cudaStream_t, cudaStreamCaptureMode)
ALWAYS_OK(cudaStreamEndCapture, cudaStream_t, cudaGraph_t *)
ALWAYS_OK(cudaGraphInstantiate, cudaGraphExec_t *, cudaGraph_t, unsigned long long)
ALWAYS_OK(cudaGraphLaunch, cudaGraphExec_t, cudaStream_t)
ALWAYS_OK(cudaGraphDestroy, cudaGraph_t)
ALWAYS_OK(cudaGraphExecDestroy, cudaGraphExec_t)
ALWAYS_OK(cudaLaunchHostFunc, cudaStream_t, cudaHostFn_t, void *)

}  // extern "C"
