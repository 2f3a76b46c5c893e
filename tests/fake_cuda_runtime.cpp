// A CUDA runtime without a GPU, for tests of the library's host code: memory is
// host memory, copies are copies, kernels do not run, and what the library asks
// of the runtime is checked: a launch needs its kernel's limit of dynamic shared
// memory raised on the current device. The serve kernel alone is stood in for:
// fake_run_serve runs the queued ones, warp after warp, over the ring that the
// server gave them. Linked with the library's objects in the runtime's place.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

// device intrinsics that inline functions of the headers name
inline size_t __cvta_generic_to_shared(const void *) { return 0; }
inline long long clock64() { return 0; }
inline int atomicExch(int *, int) { return 0; }

#include "ann_internal.cuh"
#include "serve_take.cuh"

namespace {

constexpr size_t kOptin = 232448, kDefaultLimit = 49152;
thread_local int device = 0;
thread_local cudaError_t last = cudaSuccess;
std::map<std::pair<int, const void *>, size_t> limits;
std::map<const void *, std::string> names;
bool in_hook = false;

struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t stream;
};
thread_local std::vector<Config> pushed;

struct Serve {
    ann::ServeRing ring;
    uint32_t warps;
};
std::vector<Serve> queued;

cudaError_t result(cudaError_t e)
{
    if (e != cudaSuccess) last = e;
    return e;
}

size_t limit(const void *f)
{
    const auto it = limits.find({device, f});
    return it == limits.end() ? kDefaultLimit : it->second;
}

struct HostCounts {
    static constexpr uint32_t kLooks = 4;
    unsigned long long *c;
    unsigned long long load(uint32_t i) { return c[i]; }
    unsigned long long add(uint32_t i, unsigned long long x) { return std::exchange(c[i], c[i] + x); }
    unsigned long long max(uint32_t i, unsigned long long x) { return std::exchange(c[i], std::max(c[i], x)); }
    void fence() {}
    void gave_up() {}
};

void *handle() { return std::malloc(8); }

}  // namespace

extern "C" {

int fake_busy = 0;                       // cudaStreamQuery's answer
int fake_fail_launches = 0;              // launches to refuse
unsigned long long fake_launches = 0, fake_pools = 0, fake_temporaries = 0, fake_trims = 0, fake_pool_keep = 0;
int fake_no_temporaries = 0;             // refuse allocations from a pool
int fake_no_memory = 0;                  // refuse cudaMalloc
int fake_capturing = 0;                  // cudaStreamIsCapturing's answer
void (*fake_after_limit)(void) = nullptr;   // called after each cudaFuncSetAttribute outside the hook itself

void fake_set_device(int d) { device = d; }

void fake_run_serve()
{
    for (const Serve &s : queued) {
        const ann::ServeRing &r = s.ring;
        for (uint32_t w = 0; w < s.warps; ++w) {
            HostCounts c{r.counters};
            ann::serve_publish(c, ann::serve_tail(r.tail, r.live ? *r.live : 0));
            unsigned long long h = 0;
            for (uint32_t served = 0; served < r.per_warp && ann::serve_take(c, &h); ++served) {
                const uint32_t ri = r.slot_req[h % r.cap];
                if (++r.done[ri] == r.reqs[ri].nq) {
                    r.done[ri] = 0;
                    r.flags[r.reqs[ri].flag] = 1;
                }
            }
        }
    }
    queued.clear();
}

// ------------------------------------------------------------ kernels
void **__cudaRegisterFatBinary(void *) { return (void **)handle(); }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
void __cudaRegisterFunction(void **, const char *host, char *, const char *name, int, void *, void *, void *, void *,
                            int *)
{
    names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t stream)
{
    pushed.push_back(Config{grid, block, smem, stream});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3 *grid, dim3 *block, size_t *smem, void *stream)
{
    const Config c = pushed.back();
    pushed.pop_back();
    *grid = c.grid;
    *block = c.block;
    *smem = c.smem;
    *(cudaStream_t *)stream = c.stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t *k, const void *f)
{
    *k = (cudaKernel_t)f;
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void **args, size_t smem, cudaStream_t)
{
    const void *f = (const void *)k;
    if (fake_fail_launches > 0) {
        --fake_fail_launches;
        return result(cudaErrorLaunchOutOfResources);
    }
    if (smem > limit(f) || grid.x == 0) return result(cudaErrorInvalidValue);
    ++fake_launches;
    if (names[f].find("serve_kernel") != std::string::npos)
        queued.push_back(Serve{*(const ann::ServeRing *)args[1], grid.x * block.x / 32});
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *f, void **args)
{
    return __cudaLaunchKernel((cudaKernel_t)f, c->gridDim, c->blockDim, args, c->dynamicSmemBytes, c->stream);
}
cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v)
{
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaSuccess;
    if ((size_t)v > kOptin) return result(cudaErrorInvalidValue);
    limits[{device, f}] = (size_t)v;
    if (fake_after_limit && !in_hook) {
        in_hook = true;
        fake_after_limit();
        in_hook = false;
    }
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int, size_t smem, unsigned)
{
    *n = smem > limit(f) ? 0 : (int)std::min<size_t>(4, kOptin / (smem + 1024));
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *)
{
    *n = 76;
    return cudaSuccess;
}

// ------------------------------------------------------------ devices, memory
cudaError_t cudaGetDeviceCount(int *n)
{
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int *d)
{
    *d = device;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d)
{
    device = d;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int)
{
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? (int)kOptin : 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetStreamPriorityRange(int *lo, int *hi)
{
    *lo = *hi = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return std::exchange(last, cudaSuccess); }
const char *cudaGetErrorString(cudaError_t) { return "an error of the stand-in runtime"; }
cudaError_t cudaMalloc(void **p, size_t n)
{
    *p = fake_no_memory ? nullptr : std::calloc(1, n + 256);
    return *p ? cudaSuccess : result(cudaErrorMemoryAllocation);
}
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
struct CUmemPoolHandle_st {
    int device;
    unsigned long long keep;
};
cudaError_t cudaMemPoolCreate(cudaMemPool_t *pool, const cudaMemPoolProps *props)
{
    ++fake_pools;
    *pool = new CUmemPoolHandle_st{props->location.id, 0};
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t pool, cudaMemPoolAttr a, void *value)
{
    if (a == cudaMemPoolAttrReleaseThreshold) pool->keep = fake_pool_keep = *(unsigned long long *)value;
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void **p, size_t n, cudaMemPool_t pool, cudaStream_t)
{
    if (fake_no_temporaries || pool->device != device) return result(cudaErrorMemoryAllocation);
    ++fake_temporaries;
    return cudaMalloc(p, n);
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t)
{
    ++fake_trims;
    return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s)
{
    *s = fake_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned)
{
    *d = h;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p)
{
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind)
{
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind k, cudaStream_t) { return cudaMemcpy(d, s, n, k); }
cudaError_t cudaMemcpy2D(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind)
{
    for (size_t i = 0; i < h; ++i) std::memcpy((char *)d + i * dp, (const char *)s + i * sp, w);
    return cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind k,
                              cudaStream_t)
{
    return cudaMemcpy2D(d, dp, s, sp, w, h, k);
}
cudaError_t cudaMemset(void *p, int v, size_t n)
{
    std::memset(p, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaGetSymbolAddress(void **p, const void *s)
{
    *p = (void *)s;
    return cudaSuccess;
}

// ------------------------------------------------------------ streams, events
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned)
{
    *s = (cudaStream_t)handle();
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t *s, unsigned, int) { return cudaStreamCreateWithFlags(s, 0); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return cudaFree(s); }
cudaError_t cudaStreamQuery(cudaStream_t) { return fake_busy ? cudaErrorNotReady : cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned)
{
    *e = (cudaEvent_t)handle();
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t e) { return cudaFree(e); }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }

static CUresult encode(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                       const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                       CUtensorMapL2promotion, CUtensorMapFloatOOBfill)
{
    return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q)
{
    *fn = (void *)encode;
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}

}  // extern "C"
