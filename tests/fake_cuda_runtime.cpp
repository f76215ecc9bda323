// A CUDA runtime on the host for tests of the library's host code: memory is host memory, kernels
// are only written down.  It knows two devices, and, as the real runtime does, it refuses a launch
// with more than 48 KB of dynamic shared memory unless the limit was raised for that kernel on the
// current device.
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

#include <cuda_runtime_api.h>

namespace {
struct Launch {
    std::string name;
    dim3 grid, block;
    size_t shared;
    bool chained;
};
int g_device = 0, g_failing_attributes = 0;
std::map<const void *, std::string> &names()
{
    static std::map<const void *, std::string> m;
    return m;
}
std::map<std::pair<int, const void *>, size_t> g_limit;
std::vector<Launch> g_launches;
struct Config {
    dim3 grid, block;
    size_t shared;
    void *stream;
};
std::vector<Config> g_config;

cudaError_t launch(const void *fn, dim3 grid, dim3 block, size_t shared, bool chained)
{
    const auto it = g_limit.find({g_device, fn});
    const size_t limit = it == g_limit.end() ? size_t{48} << 10 : it->second;
    if (shared > limit) return cudaErrorInvalidValue;
    g_launches.push_back(Launch{names()[fn], grid, block, shared, chained});
    return cudaSuccess;
}
}  // namespace

#define API extern "C" __attribute__((visibility("default")))

API void fake_set_device(int d) { g_device = d; }
API void fake_fail_attributes(int n) { g_failing_attributes = n; }
API void fake_clear() { g_launches.clear(); }
API int fake_launches() { return static_cast<int>(g_launches.size()); }
API const char *fake_launch(int k, unsigned *grid, unsigned *block, unsigned *shared, int *chained)
{
    const Launch &l = g_launches.at(static_cast<size_t>(k));
    grid[0] = l.grid.x;
    grid[1] = l.grid.y;
    grid[2] = l.grid.z;
    *block = l.block.x;
    *shared = static_cast<unsigned>(l.shared);
    *chained = l.chained ? 1 : 0;
    return l.name.c_str();
}

extern "C" {
void **__cudaRegisterFatBinary(void *) { return static_cast<void **>(std::calloc(1, 8)); }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, void *,
                            void *, void *, void *, int *)
{
    names()[host] = name;
}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t shared, void *stream)
{
    g_config.push_back(Config{grid, block, shared, stream});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *shared, void *stream)
{
    const Config c = g_config.back();
    g_config.pop_back();
    *grid = c.grid;
    *block = c.block;
    *shared = c.shared;
    *static_cast<void **>(stream) = c.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *fn)
{
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void *>(fn));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **, size_t shared,
                               cudaStream_t)
{
    return launch(reinterpret_cast<const void *>(k), grid, block, shared, false);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *fn, void **)
{
    bool chained = false;
    for (unsigned k = 0; k < c->numAttrs; ++k)
        chained |= c->attrs[k].id == cudaLaunchAttributeProgrammaticStreamSerialization &&
                   c->attrs[k].val.programmaticStreamSerializationAllowed;
    return launch(fn, c->gridDim, c->blockDim, c->dynamicSmemBytes, chained);
}
cudaError_t cudaFuncSetAttribute(const void *fn, cudaFuncAttribute attr, int value)
{
    if (g_failing_attributes > 0) {
        --g_failing_attributes;
        return cudaErrorUnknown;
    }
    if (attr == cudaFuncAttributeMaxDynamicSharedMemorySize)
        g_limit[{g_device, fn}] = static_cast<size_t>(value);
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int,
                                                                   size_t, unsigned)
{
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d)
{
    *d = g_device;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int)
{
    *v = 152;   // the one attribute the library asks for: multiprocessors
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "none" : "fake error"; }
cudaError_t cudaGetSymbolAddress(void **p, const void *)
{
    static void *mem = std::calloc(1, size_t{64} << 20);
    *p = mem;
    return cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t n)
{
    *p = std::calloc(1, n);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void *p)
{
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemset(void *p, int v, size_t n)
{
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind)
{
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t)
{
    return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemcpy2D(void *, size_t, const void *, size_t, size_t, size_t, cudaMemcpyKind)
{
    return cudaErrorNotSupported;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e)
{
    *e = reinterpret_cast<cudaEvent_t>(std::malloc(1));
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e)
{
    std::free(e);
    return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t)
{
    *ms = 1.0f;
    return cudaSuccess;
}
}
