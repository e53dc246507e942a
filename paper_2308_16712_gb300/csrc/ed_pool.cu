// ed_pool.cu -- a library-private, stream-ordered device memory pool for the
// arrays the library allocates itself: the solvers' work vectors, the basis
// build's temporaries and the large arrays of a basis.  cudaMalloc / cudaFree
// of gigabytes take milliseconds and synchronise the device; memory freed back
// to this pool is kept (up to a release threshold, 1/16 of the device memory,
// applied at synchronisation points) and handed out again by
// the next call without either cost.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <tuple>

#include "ed_kernels.cuh"

namespace edk {
namespace {

constexpr int kMaxDevices = 64;
std::mutex g_pool_mutex;
cudaMemPool_t g_pools[kMaxDevices] = {};

cudaError_t device_pool(cudaMemPool_t *out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    if (dev < 0 || dev >= kMaxDevices)
        return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    if (!g_pools[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        if ((e = cudaMemPoolCreate(&p, &props)) != cudaSuccess)
            return e;
        size_t free_b = 0, total_b = 0;
        cudaMemGetInfo(&free_b, &total_b);
        uint64_t keep = total_b / 16;
        if ((e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) {
            cudaMemPoolDestroy(p);
            return e;
        }
        g_pools[dev] = p;
    }
    *out = g_pools[dev];
    return cudaSuccess;
}

}  // namespace

cudaError_t ws_alloc(void **p, size_t bytes, cudaStream_t s)
{
    cudaMemPool_t pool;
    cudaError_t e = device_pool(&pool);
    if (e != cudaSuccess)
        return e;
    return cudaMallocFromPoolAsync(p, std::max<size_t>(bytes, 1), pool, s);
}

namespace {
std::atomic<uint64_t> g_optional_limit{~0ull};
}  // namespace

cudaError_t ws_alloc_optional(void **p, size_t bytes, cudaStream_t s)
{
    *p = nullptr;
    if (bytes > g_optional_limit.load(std::memory_order_relaxed))
        return cudaErrorMemoryAllocation;
    const cudaError_t e = ws_alloc(p, bytes, s);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        *p = nullptr;
    }
    return e;
}

cudaError_t ws_free(void *p, cudaStream_t s)
{
    return p ? cudaFreeAsync(p, s) : cudaSuccess;
}

size_t ws_cached_bytes()
{
    cudaMemPool_t pool;
    if (device_pool(&pool) != cudaSuccess)
        return 0;
    uint64_t reserved = 0, used = 0;
    if (cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReservedMemCurrent, &reserved) != cudaSuccess ||
        cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess)
        return 0;
    return reserved > used ? (size_t)(reserved - used) : 0;
}

cudaError_t kernel_occupancy(const void *kern, int threads, size_t smem, int *sms, int *per_sm)
{
    static std::mutex m;
    static std::map<std::tuple<int, const void *, size_t>, std::pair<int, int>> known;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess)
        return e;
    std::lock_guard<std::mutex> lock(m);
    const auto key = std::make_tuple(dev, kern, smem);
    auto it = known.find(key);
    if (it == known.end()) {
        int n = 0, k = 0, limit = 0;
        // the limit only ever grows, so that launches of other sizes in flight keep theirs
        cudaFuncAttributes fa;
        if ((e = cudaFuncGetAttributes(&fa, kern)) != cudaSuccess)
            return e;
        limit = std::max(fa.maxDynamicSharedSizeBytes, (int)smem);
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, limit)) != cudaSuccess ||
            (e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
            (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&k, kern, threads, smem)) != cudaSuccess)
            return e;
        it = known.emplace(key, std::make_pair(n, k)).first;
    }
    *sms = it->second.first;
    *per_sm = it->second.second;
    return cudaSuccess;
}

}  // namespace edk

// Test hook: later requests for work memory that the library can do without are
// refused above this many bytes, as if the device had none.
extern "C" void edx_optional_memory(uint64_t bytes)
{
    edk::g_optional_limit.store(bytes, std::memory_order_relaxed);
}

extern "C" ed_status ed_release_cached_memory(void)
{
    std::lock_guard<std::mutex> lock(edk::g_pool_mutex);
    for (cudaMemPool_t p : edk::g_pools)
        if (p && cudaMemPoolTrimTo(p, 0) != cudaSuccess)
            return ED_ERR_CUDA;
    return ED_OK;
}
