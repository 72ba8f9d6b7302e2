// A CUDA runtime for host-side tests, preloaded before the library in a process
// without a GPU.  Device memory is host memory, kernels do nothing, and every
// copy, set and launch is checked the way the device would:
//  - a copy's or set's device range lies inside one live allocation,
//  - a launch has blocks, and its dynamic shared memory is within its kernel's limit,
//  - the limit of a kernel is not lowered (it belongs to the process, so
//    lowering it refuses another thread's launch in between).
// fake_reset(k) clears the records and makes the k-th allocation from then on
// fail (k < 0: none); fake_report gives what was found.
#include <cuda_runtime.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>

namespace {
std::map<char *, size_t> live;
std::map<const void *, int> limit;
std::string found;
long countdown = -1, failed = 0, pinned = 0, waits = 0;
cudaError_t last = cudaSuccess;

cudaError_t keep(cudaError_t e)
{
    if (e != cudaSuccess) last = e;
    return e;
}
void check(const char *what, const void *p, size_t n)
{
    auto it = live.upper_bound((char *)p);
    if (it == live.begin()) return;                    // not device memory
    --it;
    const size_t at = (char *)p - it->first;
    if (at < it->second && at + n > it->second)
        found += std::string(what) + " " + std::to_string(at + n - it->second) +
                 " bytes past an allocation of " + std::to_string(it->second) + "; ";
}
cudaError_t launch(const void *f, dim3 grid, size_t smem)
{
    if (!grid.x || !grid.y || !grid.z) return keep(cudaErrorInvalidConfiguration);
    const auto it = limit.find(f);
    const size_t most = it == limit.end() ? 48 * 1024 : it->second;
    if (smem <= most) return cudaSuccess;
    found += "a launch with " + std::to_string(smem) + " bytes of shared memory, limit " +
             std::to_string(most) + "; ";
    return keep(cudaErrorInvalidValue);
}
cudaError_t copy(void *d, const void *s, size_t n)
{
    check("copy into", d, n);
    check("copy from", s, n);
    if (found.empty()) memcpy(d, s, n);
    return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_reset(long k) { found.clear(); countdown = k; failed = 0; }
const char *fake_report() { return found.c_str(); }
long fake_live() { return (long)live.size(); }
long fake_failed() { return failed; }
long fake_pinned() { return pinned; }
long fake_waits() { return waits; }

cudaError_t cudaMalloc(void **p, size_t n)
{
    if (countdown >= 0 && countdown-- == 0) {
        ++failed;
        return keep(cudaErrorMemoryAllocation);
    }
    *p = calloc(1, n + 1);
    live[(char *)*p] = n;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    if (!p) return cudaSuccess;
    if (!live.erase((char *)p)) found += "free of an unknown pointer; ";
    else free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned)
{
    ++pinned;
    *p = malloc(n);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemGetInfo(size_t *f, size_t *t) { *f = *t = (size_t)1 << 38; return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { return copy(d, s, n); }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { return copy(d, s, n); }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t)
{
    check("set of", d, n);
    if (found.empty()) memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v)
{
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaSuccess;
    if (limit.count(f) && v < limit[f])
        found += "a kernel's shared-memory limit lowered from " + std::to_string(limit[f]) +
                 " to " + std::to_string(v) + "; ";
    limit[f] = v;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **)
{
    return launch(f, c->gridDim, c->dynamicSmemBytes);
}
cudaError_t cudaLaunchCooperativeKernel(const void *f, dim3 grid, dim3, void **, size_t smem, cudaStream_t)
{
    return launch(f, grid, smem);
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void **, size_t smem, cudaStream_t)
{
    return launch((const void *)k, grid, smem);
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) { memset(a, 0, sizeof *a); return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned)
{
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *)
{
    *n = 7;
    return cudaSuccess;
}
cudaError_t cudaGetLastError()
{
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void **, const void *) { return cudaErrorInvalidValue; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { ++waits; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *) { return cudaErrorNotSupported; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
}
