// The memory of ray contexts. A context's state is one device block and one
// pinned word block; released blocks are kept for the next context of about the
// same size, because allocating and freeing them cost more than tracing a small
// bundle (ten allocations and frees: 0.5 ms for 128^2 rays, 1.1 ms for 2048^2,
// against 50 us for a 64-cell step of 128^2 rays).
//
// Bounds: at most kMostBytes and kMostBlocks are kept, the oldest are freed
// first, a block larger than kMostBytes is freed at once, an allocation of the
// library that fails empties the pool and is tried again, and rr_release_cached
// empties it on demand. A block is handed out on the device it was allocated on,
// to one holder at a time (a mutex guards the list), and is given back only after
// the device has finished with it, so any stream and thread may use it next. A
// block whose CUDA context is gone (cudaDeviceReset) went with it: it is neither
// handed out nor freed.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <mutex>

#include "rr_internal.h"

namespace rr {
namespace {

constexpr size_t kMostBytes = (size_t)1 << 30;
constexpr size_t kMostBlocks = 64;

// The kept blocks, oldest first. An array: a call that gives memory back may
// not fail for want of memory.
struct List {
    Block b[kMostBlocks];
    size_t n = 0;
    Block remove(size_t i)
    {
        const Block r = b[i];
        for (--n; i < n; ++i) b[i] = b[i + 1];
        return r;
    }
};

std::mutex g_mutex;
List g_kept;

// The number of the current CUDA context, made current for device dev where the
// thread has none (numbers are not used again; 0: the driver tells none).
unsigned long long context_id(int dev)
{
    static const PFN_cuCtxGetId_v12000 get = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q);
        return reinterpret_cast<PFN_cuCtxGetId_v12000>(e == cudaSuccess && q == cudaDriverEntryPointSuccess ? p : nullptr);
    }();
    unsigned long long id = 0;
    if (!get || get(nullptr, &id) == CUDA_SUCCESS) return id;
    return cudaSetDevice(dev) == cudaSuccess && get(nullptr, &id) == CUDA_SUCCESS ? id : 0;
}

void release(const Block& b)
{
    int dev = b.device;
    cudaGetDevice(&dev);
    if (dev != b.device) cudaSetDevice(b.device);
    if (context_id(b.device) == b.context) {
        cudaFree(b.dev);
        cudaFreeHost(b.host);
    }
    if (dev != b.device) cudaSetDevice(dev);
}

}  // namespace

void pool_clear()
{
    List all;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        all = g_kept;
        g_kept.n = 0;
    }
    for (size_t i = 0; i < all.n; ++i) release(all.b[i]);
}

namespace {

template <class F>
cudaError_t alloc_again(F alloc)
{
    cudaError_t e = alloc();
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();   // (or the next launch would report it)
    pool_clear();
    e = alloc();
    if (e == cudaErrorMemoryAllocation) cudaGetLastError();
    return e;
}

}  // namespace

cudaError_t device_alloc(void** p, size_t bytes)
{
    return alloc_again([&] { return cudaMalloc(p, bytes); });
}

cudaError_t pinned_alloc(void** p, size_t bytes)
{
    return alloc_again([&] { return cudaMallocHost(p, bytes); });
}

cudaError_t pool_take(size_t bytes, Block* out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long context = context_id(dev);
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        const List& v = g_kept;
        size_t best = v.n;
        // the smallest that fits and wastes no more than a quarter (or 1 MB)
        for (size_t i = 0; i < v.n; ++i)
            if (v.b[i].device == dev && v.b[i].context == context && v.b[i].bytes >= bytes &&
                v.b[i].bytes - bytes <= bytes / 4 + ((size_t)1 << 20) &&
                (best == v.n || v.b[i].bytes < v.b[best].bytes))
                best = i;
        if (best < v.n) {
            *out = g_kept.remove(best);
            return cudaSuccess;
        }
    }
    Block b;
    b.bytes = bytes;
    b.device = dev;
    b.context = context;
    e = device_alloc(&b.dev, bytes);
    if (e != cudaSuccess) return e;
    e = pinned_alloc(reinterpret_cast<void**>(&b.host), sizeof(HostWords));
    if (e != cudaSuccess) {
        cudaFree(b.dev);
        return e;
    }
    *out = b;
    return cudaSuccess;
}

void pool_give(const Block& b, bool idle)
{
    if (!b.dev) return;
    if (!idle || b.bytes > kMostBytes || context_id(b.device) != b.context) {
        release(b);
        return;
    }
    List old;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        size_t total = b.bytes;
        for (size_t i = 0; i < g_kept.n; ++i) total += g_kept.b[i].bytes;
        while (g_kept.n && (total > kMostBytes || g_kept.n == kMostBlocks)) {
            total -= g_kept.b[0].bytes;
            old.b[old.n++] = g_kept.remove(0);
        }
        g_kept.b[g_kept.n++] = b;
    }
    for (size_t i = 0; i < old.n; ++i) release(old.b[i]);
}

}  // namespace rr

extern "C" rr_status rr_release_cached(void)
{
    rr::pool_clear();
    return RR_OK;
}
