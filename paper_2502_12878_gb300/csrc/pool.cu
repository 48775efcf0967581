// The library's memory pool (pool.cuh).  Host code on the runtime API only, and the
// driver's context functions by their entry points, so that it can be compiled
// against a fake of both.
#include <string.h>

#include <mutex>

#include "pool.cuh"

namespace rbffd {

// A pool lives as long as its device's primary context: after a cudaDeviceReset
// the context's id is another one, and a new pool is made (the old one went with
// its context).  A thread whose caller has made a context of its own current is
// left in it, and gets its memory from the device's default pool.
namespace {
struct Pools {
    static constexpr int MAX_DEV = 64;
    std::mutex mu;
    cudaMemPool_t pool[MAX_DEV] = {};
    unsigned long long ctx[MAX_DEV] = {};
    // driver functions (CUcontext as void*, CUdevice as int)
    int (*ctx_id)(void*, unsigned long long*) = nullptr;
    int (*ctx_current)(void**) = nullptr;
    int (*device_get)(int*, int) = nullptr;
    int (*primary_state)(int, unsigned*, int*) = nullptr;
    int (*primary_retain)(void**, int) = nullptr;
    int (*primary_release)(int) = nullptr;
    bool looked = false, found_all = false;
    ~Pools() {
        for (int d = 0; d < MAX_DEV; ++d)
            if (pool[d]) cudaMemPoolDestroy(pool[d]);   // (an error when CUDA has shut down)
    }
    template <class F>
    static bool entry(const char* name, unsigned version, F** fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion(name, &p, version, cudaEnableDefault, &found) !=
                cudaSuccess ||
            found != cudaDriverEntryPointSuccess)
            return false;
        *fn = reinterpret_cast<F*>(p);
        return true;
    }
    void look() {
        looked = true;
        found_all = entry("cuCtxGetId", 12000, &ctx_id) &&
                    entry("cuCtxGetCurrent", 4000, &ctx_current) &&
                    entry("cuDeviceGet", 2000, &device_get) &&
                    entry("cuDevicePrimaryCtxGetState", 7000, &primary_state) &&
                    entry("cuDevicePrimaryCtxRetain", 7000, &primary_retain) &&
                    entry("cuDevicePrimaryCtxRelease", 11000, &primary_release);
    }
    // whether the current context is device dev's primary one
    bool in_primary(int dev) {
        void *cur = nullptr, *primary = nullptr;
        int cu = 0, active = 0;
        unsigned flags = 0;
        if (ctx_current(&cur) != 0 || device_get(&cu, dev) != 0 ||
            primary_state(cu, &flags, &active) != 0 || !active || primary_retain(&primary, cu) != 0)
            return false;
        primary_release(cu);
        return cur == primary;
    }
    // the current device's pool; null where there can be none
    cudaMemPool_t get() {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEV) return nullptr;
        std::lock_guard<std::mutex> lock(mu);
        if (!looked) look();
        if (!found_all) return nullptr;
        // a thread without a context gets the device's primary one, as its first
        // runtime call would give it
        unsigned long long id = 0;
        void* cur = nullptr;
        if (ctx_current(&cur) != 0) cur = nullptr;   // (the driver is not initialised yet)
        if (!cur && cudaSetDevice(dev) != cudaSuccess) return nullptr;
        if (ctx_id(nullptr, &id) != 0) return nullptr;
        if (pool[dev] && ctx[dev] == id) return pool[dev];   // (ids are not used again)
        if (!in_primary(dev)) return nullptr;
        cudaMemPoolProps props;
        memset(&props, 0, sizeof(props));
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t made = nullptr;
        unsigned long long keep = POOL_KEEP;
        if (cudaMemPoolCreate(&made, &props) != cudaSuccess ||
            cudaMemPoolSetAttribute(made, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        pool[dev] = made;
        ctx[dev] = id;
        return made;
    }
};
Pools g_pools;
}  // namespace

cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t s) {
    cudaMemPool_t pool = g_pools.get();
    if (!pool) return cudaMallocAsync(p, bytes, s);
    cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    if (e == cudaErrorMemoryAllocation) {   // with what the pool keeps given back
        cudaGetLastError();
        cudaStreamSynchronize(s);
        cudaMemPoolTrimTo(pool, 0);
        e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    }
    return e;
}

void pool_free(void* const* p, int n) {
    int first = 0, cur = 0;
    while (first < n && !p[first]) ++first;
    if (first == n) return;
    cudaPointerAttributes a;
    const bool known = cudaGetDevice(&cur) == cudaSuccess &&
                       cudaPointerGetAttributes(&a, p[first]) == cudaSuccess;
    if (!known) cudaGetLastError();
    const bool other = known && a.device != cur;
    if (other) cudaSetDevice(a.device);
    cudaDeviceSynchronize();
    for (int i = first; i < n; ++i)
        if (p[i]) cudaFreeAsync(p[i], cudaStreamPerThread);
    // the pool gives back what it need not keep at a synchronisation, and not before
    cudaStreamSynchronize(cudaStreamPerThread);
    if (other) cudaSetDevice(cur);
}

}  // namespace rbffd
