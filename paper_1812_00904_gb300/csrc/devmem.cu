// Device memory of plans and of calls that need scratch: a private memory pool per device.
//
// cudaMalloc and cudaFree take about 100 us each on this machine (a plan makes eight, a CGLS call
// two: 0.8 of the 2.4 ms of ingesting 10M triples, 0.2 of the 1.0 ms of a short CGLS run).  The
// pool keeps up to POOL_KEEP bytes of freed memory for the next plan and gives everything beyond
// back to the device at its next synchronisation; when an allocation of the library fails, whether
// from the pool or beside it, it gives all of it back and tries again, and spmv_release_memory gives
// it back for others.  The allocations and frees go through a stream of the pool's own: memory is
// handed out after that stream was waited for, so it can be used on any stream, and the caller
// frees memory only when no work that uses it is pending.  Every call is safe from any thread.
//
// Blocks of more than half of what the pool keeps bypass it: a pool grows at 0.87 us per MB and gives
// back at 2.5 (256 MB: 228 us and 1.0 ms; 2 GB: 1.7 and 13 ms), cudaMalloc and cudaFree take 56 + 197
// us for 256 MB and 0.1 + 1.4 ms for 2 GB, while a kept block costs 2 us.  (A bank-ordered plan of
// 200M nonzeros: 14.5 ms with its 2.4 GB from the pool, 13.0 without.)
#include <cuda_runtime.h>

#include <mutex>
#include <unordered_map>
#include <unordered_set>

#include "plan_impl.h"

namespace gbk {
namespace {

constexpr uint64_t POOL_KEEP = 512ull << 20;
constexpr size_t POOL_MOST = POOL_KEEP / 2;  // bytes of a block from the pool

struct DevicePool {
    std::once_flag once;
    cudaMemPool_t pool = nullptr;  // NULL: no pool could be made, plain allocations
    cudaStream_t stream = nullptr;
};
DevicePool g_pools[MAX_DEVICES];

std::mutex g_large_mu;
// the blocks that bypassed the pool (never destroyed: plans may be freed while the process ends)
std::unordered_set<void *> &g_large = *new std::unordered_set<void *>;
// pooled blocks freed while they might still be in use, by device (under g_large_mu)
std::unordered_multimap<int, void *> &g_late = *new std::unordered_multimap<int, void *>;

DevicePool &pool_of(int device) {
    DevicePool &P = g_pools[device];
    std::call_once(P.once, [&] {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = device;
        cudaMemPool_t pool = nullptr;
        cudaStream_t st = nullptr;
        uint64_t keep = POOL_KEEP;
        if (cudaMemPoolCreate(&pool, &props) == cudaSuccess &&
            cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) == cudaSuccess &&
            cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) == cudaSuccess) {
            P.pool = pool;
            P.stream = st;
        } else {
            cudaGetLastError();
            if (pool) cudaMemPoolDestroy(pool);
        }
    });
    return P;
}

}  // namespace

cudaError_t dev_release() {
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    if (device < 0 || device >= MAX_DEVICES) return cudaErrorInvalidDevice;
    DevicePool &P = pool_of(device);
    if (!P.pool) return cudaSuccess;
    e = cudaStreamSynchronize(P.stream);
    return e == cudaSuccess ? cudaMemPoolTrimTo(P.pool, 0) : e;
}

cudaError_t dev_malloc(void **p, size_t bytes) {
    *p = nullptr;
    cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaErrorMemoryAllocation) {  // what the pool keeps may make room
        cudaGetLastError();
        *p = nullptr;
        dev_release();
        e = cudaMalloc(p, bytes);
    }
    if (e != cudaSuccess) *p = nullptr;
    return e;
}

cudaError_t dev_alloc(void **p, size_t bytes) {
    *p = nullptr;
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    if (device < 0 || device >= MAX_DEVICES) return cudaErrorInvalidDevice;
    DevicePool &P = pool_of(device);
    if (!P.pool) return cudaMalloc(p, bytes);
    if (bytes > POOL_MOST) {
        e = dev_malloc(p, bytes);
        if (e != cudaSuccess) return e;
        std::lock_guard<std::mutex> lk(g_large_mu);
        g_large.insert(*p);
        return cudaSuccess;
    }
    for (int attempt = 0; attempt < 2; ++attempt) {
        e = cudaMallocFromPoolAsync(p, bytes, P.pool, P.stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(P.stream);
        if (e != cudaErrorMemoryAllocation) break;
        cudaGetLastError();
        *p = nullptr;
        if (attempt == 0) dev_release();
    }
    return e;
}

void dev_free(void *p, int device, bool idle) {
    if (!p) return;
    bool large;
    {
        std::lock_guard<std::mutex> lk(g_large_mu);
        large = g_large.erase(p) != 0;
    }
    if (!large && device >= 0 && device < MAX_DEVICES && g_pools[device].pool) {
        // (cudaFree waits for the device by itself, the pool for nothing: memory that may still be in use
        // must not go back to it yet)
        if (idle) {
            cudaFreeAsync(p, g_pools[device].stream);
        } else {
            std::lock_guard<std::mutex> lk(g_large_mu);
            g_late.emplace(device, p);
        }
    } else {
        cudaFree(p);
    }
}

void dev_free_late(int device) {
    std::lock_guard<std::mutex> lk(g_large_mu);
    const auto late = g_late.equal_range(device);
    for (auto it = late.first; it != late.second; ++it) cudaFreeAsync(it->second, g_pools[device].stream);
    g_late.erase(late.first, late.second);
}

}  // namespace gbk
