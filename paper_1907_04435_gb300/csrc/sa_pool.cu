// sa_pool.cu -- the library's stream-ordered memory pool.
//
// Scratch (bins, masks, sort buffers) is allocated and freed on the caller's stream within
// each call, and the handles' own arrays (BVH, sun tables, sorted receivers) come from the
// same pool, freed when the handle is destroyed.  The default pool would return memory to
// the device at every synchronisation, so a repeated call would map it again each time;
// this pool keeps up to kKeep bytes reserved instead, and a handle built again (a scene
// rebuilt every step) takes memory already mapped instead of paying cudaMalloc's latency.
//
// A caller that can do with less memory goes on after a failed allocation, so one leaves no
// error behind for a later cudaGetLastError.  The bounds-checked build can be told to fail
// an allocation (sa_check_fail_alloc): how the callers are tested without exhausting a device.
#include <atomic>
#include <mutex>
#include <vector>

#include "sa_handles.cuh"

namespace sa {

namespace {
constexpr unsigned long long kKeep = 4ull << 30;
std::mutex g_pool_mu;
std::vector<cudaMemPool_t> g_pools;   // by device ordinal; null until first use
std::atomic<unsigned long long> g_n_allocs{0}, g_alloc_bytes{0};
std::atomic<int> g_fail_in{0};        // checked build: the allocation that fails, 1 the next; 0 none

// counts one allocation; true if it is the one to fail
bool planned_failure() {
#ifdef SA_CHECKED
    int n = g_fail_in.load();
    while (n > 0 && !g_fail_in.compare_exchange_weak(n, n - 1)) {}
    return n == 1;
#else
    return false;
#endif
}

cudaError_t pool_of_current_device(cudaMemPool_t* out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if ((int)g_pools.size() <= dev) g_pools.resize(dev + 1, nullptr);
    if (!g_pools[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool = nullptr;
        e = cudaMemPoolCreate(&pool, &props);
        if (e != cudaSuccess) return e;
        unsigned long long keep = kKeep;
        e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e != cudaSuccess) {
            cudaMemPoolDestroy(pool);
            return e;
        }
        g_pools[dev] = pool;
    }
    *out = g_pools[dev];
    return cudaSuccess;
}
}  // namespace

cudaError_t scratch_alloc_bytes(void** p, size_t bytes, cudaStream_t st) {
    *p = nullptr;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = pool_of_current_device(&pool);
    if (e != cudaSuccess) return e;
    g_n_allocs.fetch_add(1, std::memory_order_relaxed);
    g_alloc_bytes.fetch_add(bytes, std::memory_order_relaxed);
    if (planned_failure()) return cudaErrorMemoryAllocation;
    e = cudaMallocFromPoolAsync(p, bytes, pool, st);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

void trim_scratch() {
    cudaMemPool_t pool = nullptr;
    if (pool_of_current_device(&pool) == cudaSuccess) cudaMemPoolTrimTo(pool, 0);
}

cudaError_t device_alloc_bytes(void** p, size_t bytes) {
    *p = nullptr;
    if (planned_failure()) return cudaErrorMemoryAllocation;
    const cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

}  // namespace sa

extern "C" int32_t sa_check_fail_alloc(int32_t n) {
#ifdef SA_CHECKED
    return sa::g_fail_in.exchange(n > 0 ? n : 0);
#else
    (void)n;
    return -1;
#endif
}

extern "C" sa_status sa_scratch_stats(uint64_t* stats) {
    if (!stats) return sa::report_error(SA_ERR_INVALID_ARG, "sa_scratch_stats: stats is NULL");
    stats[0] = sa::g_n_allocs.load(std::memory_order_relaxed);
    stats[1] = sa::g_alloc_bytes.load(std::memory_order_relaxed);
    stats[2] = 0;
    stats[3] = 0;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return SA_OK;
    }
    std::lock_guard<std::mutex> lk(sa::g_pool_mu);
    if (dev < (int)sa::g_pools.size() && sa::g_pools[dev]) {
        unsigned long long v = 0;
        if (cudaMemPoolGetAttribute(sa::g_pools[dev], cudaMemPoolAttrReservedMemCurrent, &v) == cudaSuccess)
            stats[2] = v;
        if (cudaMemPoolGetAttribute(sa::g_pools[dev], cudaMemPoolAttrUsedMemHigh, &v) == cudaSuccess)
            stats[3] = v;
    }
    return SA_OK;
}
