// Memory that handles, servers and batches take when they are made and give
// back when they go: device blocks of up to kScratchKeep bytes from a
// stream-ordered pool of this library, and pinned host blocks.
//
// What bounds it: training on a small set was mostly allocation.  Of 2.6 ms
// for n = 6238 and 1.8 ms for n = 1000, create to destroy, cudaMalloc took 75
// us, two pinned blocks 110, the decision workspace 175, and freeing them 580;
// the kernels took 1.1 and 0.45 ms.  From the pool and the list the same
// requests take a few us each (with the waits that went in the same step: 2.50
// -> 1.62 ms and 1.75 -> 1.07 ms).
//
// What is kept is bounded: the pool has at most kScratchKeep bytes per device past a
// synchronisation, used and unused (the driver counts both), the list kPinnedKeep
// bytes a process.  So blocks come from the pool only while those in use stay
// within it, and from cudaMalloc beyond: a pool that has to grow past its reserve
// maps and unmaps the memory of every block (n = 6500, a second handle beside one
// of 430 MB: create 540 us, now as with cudaMalloc alone, 280).  The pool
// gives its unused memory back as soon as a larger request (device_available
// with trim, or pool_alloc) needs it, and in gabp_batch_release.  Both are safe
// with several threads; blocks are given back only after the work that used
// them has been waited for, so that any stream can take them next.
#include "common.cuh"

#include <map>
#include <mutex>

namespace gabp {
namespace {

// Above it an allocation's cost is small against the work on it, and what
// another program on the device misses stays under 0.2 % of its memory.
constexpr size_t kScratchKeep = (size_t)512 << 20;
constexpr size_t kPinnedKeep = (size_t)4 << 20;
constexpr size_t kPinnedLeast = 4096;

std::mutex g_mutex;
std::map<int, cudaMemPool_t>& pools()
{
    static auto* m = new std::map<int, cudaMemPool_t>;   // not destroyed at exit, where CUDA may be gone
    return *m;
}
std::multimap<size_t, void*>& pinned()
{
    static auto* m = new std::multimap<size_t, void*>;
    return *m;
}
size_t g_pinned_bytes = 0;

// The current device's pool; nullptr if none was made yet (make = false) or
// none can be made.
cudaMemPool_t scratch_pool(bool make)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> lock(g_mutex);
    const auto it = pools().find(dev);
    if (it != pools().end()) return it->second;
    if (!make) return nullptr;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    uint64_t keep = kScratchKeep;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    pools().emplace(dev, pool);
    return pool;
}

uint64_t pool_bytes(cudaMemPool_t pool, cudaMemPoolAttr what)
{
    uint64_t v = 0;
    if (cudaMemPoolGetAttribute(pool, what, &v) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return v;
}

size_t unused_bytes(cudaMemPool_t pool)
{
    const uint64_t reserved = pool_bytes(pool, cudaMemPoolAttrReservedMemCurrent),
                   used = pool_bytes(pool, cudaMemPoolAttrUsedMemCurrent);
    return reserved > used ? (size_t)(reserved - used) : 0;
}

size_t pinned_class(size_t bytes)
{
    size_t c = kPinnedLeast;
    while (c < bytes) c *= 2;
    return c;
}

}  // namespace

bool scratch_fits(size_t bytes) { return bytes <= kScratchKeep; }

void scratch_trim()
{
    if (cudaMemPool_t pool = scratch_pool(false)) cudaMemPoolTrimTo(pool, 0);
}

cudaError_t scratch_alloc(DevBlock* b, size_t bytes, cudaStream_t s)
{
    *b = DevBlock{};
    if (scratch_fits(bytes)) {
        const cudaMemPool_t pool = scratch_pool(true);
        if (pool && pool_bytes(pool, cudaMemPoolAttrUsedMemCurrent) + bytes <= kScratchKeep) {
            if (cudaMallocFromPoolAsync(&b->p, bytes, pool, s) == cudaSuccess) {
                b->pooled = true;
                return cudaSuccess;
            }
            cudaGetLastError();
            b->p = nullptr;
        }
    }
    cudaError_t e = cudaMalloc(&b->p, bytes);
    if (e == cudaErrorMemoryAllocation) {   // the pools' unused memory back first
        cudaGetLastError();
        size_t avail = 0;
        device_available(&avail, true);
        e = cudaMalloc(&b->p, bytes);
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        b->p = nullptr;
    }
    return e;
}

void scratch_free(DevBlock* b, cudaStream_t s)
{
    // (a pool block can be freed either way: cudaFree waits for the device)
    if (b->p && (!b->pooled || cudaFreeAsync(b->p, s) != cudaSuccess)) {
        if (b->pooled) cudaGetLastError();
        cudaFree(b->p);
    }
    *b = DevBlock{};
}

cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t s)
{
    cudaError_t e = cudaMallocAsync(p, bytes, s);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        scratch_trim();
        e = cudaMallocAsync(p, bytes, s);
    }
    return e;
}

cudaError_t pinned_alloc(void** p, size_t bytes)
{
    const size_t c = pinned_class(bytes);
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        const auto it = pinned().find(c);
        if (it != pinned().end()) {
            *p = it->second;
            pinned().erase(it);
            g_pinned_bytes -= c;
            return cudaSuccess;
        }
    }
    return cudaHostAlloc(p, c, cudaHostAllocPortable);
}

void pinned_free(void* p, size_t bytes)
{
    if (!p) return;
    const size_t c = pinned_class(bytes);
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        if (g_pinned_bytes + c <= kPinnedKeep) {
            pinned().emplace(c, p);
            g_pinned_bytes += c;
            return;
        }
    }
    cudaFreeHost(p);
}

void pinned_trim()
{
    std::lock_guard<std::mutex> lock(g_mutex);
    for (auto& kv : pinned()) cudaFreeHost(kv.second);
    pinned().clear();
    g_pinned_bytes = 0;
}

cudaError_t device_available(size_t* avail, bool trim)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    cudaMemPool_t pool;
    e = cudaDeviceGetDefaultMemPool(&pool, dev);
    if (e != cudaSuccess) return e;
    const cudaMemPool_t own = scratch_pool(false);
    if (trim) {
        e = cudaMemPoolTrimTo(pool, 0);
        if (e == cudaSuccess && own) e = cudaMemPoolTrimTo(own, 0);
        if (e != cudaSuccess) return e;
    }
    size_t free_b = 0, total_b = 0;
    e = cudaMemGetInfo(&free_b, &total_b);
    if (e != cudaSuccess) return e;
    *avail = free_b + unused_bytes(pool) + (own ? unused_bytes(own) : 0);
    return cudaSuccess;
}

}  // namespace gabp
