// fake_cudart.cpp -- the CUDA runtime calls that libsgrid makes, without a
// GPU: device memory is host memory, copies and memsets are done at once,
// kernels do not run but their launches are logged.  Linked with the library's
// own objects it shows what the host side asks of the runtime: several devices,
// a stream being recorded, refused calls.  Of a real runtime's rules it has
// those that the tests need: dynamic shared memory above 48 KB must have been
// allowed for the kernel on the current device, an empty grid is refused, a
// stream being recorded cannot be waited for, and the last error of a thread
// stays until cudaGetLastError.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>

namespace {

struct Push {
    dim3 grid, block;
    size_t smem;
    cudaStream_t s;
};
std::map<const void *, std::string> &names()
{
    static std::map<const void *, std::string> m;
    return m;
}
std::map<std::pair<int, const void *>, int> allowed;  // (device, kernel) -> dynamic shared memory
std::string launch_log;                                // "name;" per launch
thread_local Push push;
thread_local int device = 0;
thread_local cudaError_t last = cudaSuccess;
const void *recorded = nullptr;  // the stream being recorded, plus one
int refuse_attributes = 0;

cudaError_t err(cudaError_t e)
{
    if (e != cudaSuccess) last = e;
    return e;
}
const void *key(cudaStream_t s) { return (const char *)s + 1; }

cudaError_t launch(const void *f, dim3 grid, size_t smem)
{
    if (grid.x == 0) return err(cudaErrorInvalidConfiguration);
    if (smem > 49152) {
        const auto it = allowed.find({device, f});
        if (it == allowed.end() || (size_t)it->second < smem) return err(cudaErrorInvalidValue);
    }
    launch_log += names()[f] + ";";
    return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- for the tests ----
void fake_device(int d) { device = d; }
void fake_refuse_attributes(int on) { refuse_attributes = on; }
const char *fake_log() { return launch_log.c_str(); }
void fake_clear_log() { launch_log.clear(); }

// ---- what compiled kernels' host stubs call ----
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, uint3 *, uint3 *, dim3 *, dim3 *, int *)
{
    names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st *s)
{
    push = {grid, block, smem, s};
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *s)
{
    *grid = push.grid;
    *block = push.block;
    *smem = push.smem;
    *(cudaStream_t *)s = push.s;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f)
{
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **, size_t smem, cudaStream_t)
{
    return launch((const void *)k, grid, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **)
{
    return launch(f, c->gridDim, c->dynamicSmemBytes);
}

// ---- devices, kernels, errors ----
cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, enum cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *f, enum cudaFuncAttribute a, int v)
{
    if (refuse_attributes) return err(cudaErrorInvalidValue);
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) allowed[{device, f}] = v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) { *n = 2; return cudaSuccess; }
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaPeekAtLastError() { return last; }
const char *cudaGetErrorString(cudaError_t) { return "refused by the fake runtime"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **, unsigned, unsigned long long, enum cudaDriverEntryPointQueryResult *) { return err(cudaErrorNotSupported); }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return err(cudaErrorInvalidValue); }

// ---- memory ----
cudaError_t cudaMalloc(void **p, size_t n) { *p = std::aligned_alloc(256, (n + 255) / 256 * 256); return *p ? cudaSuccess : err(cudaErrorMemoryAllocation); }
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, enum cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, enum cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { *f = *t = size_t(1) << 34; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes *, const void *) { return err(cudaErrorInvalidValue); }

// ---- streams, events, recordings ----
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return recorded == key(s) ? err(cudaErrorStreamCaptureUnsupported) : cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = (cudaStream_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus *st)
{
    *st = recorded == key(s) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, enum cudaStreamCaptureMode) { recorded = key(s); return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { recorded = nullptr; *g = (cudaGraph_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) { *e = (cudaGraphExec_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { std::free(g); return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = (cudaEvent_t)std::malloc(1); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }

}  // extern "C"
