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
// the device has finished with it, so any stream and thread may use it next.
#include <mutex>
#include <vector>

#include "rr_internal.h"

namespace rr {
namespace {

constexpr size_t kMostBytes = (size_t)1 << 30;
constexpr size_t kMostBlocks = 64;

std::mutex g_mutex;
std::vector<Block>& kept()
{
    static std::vector<Block>* v = new std::vector<Block>();   // never destroyed: outlives every context
    return *v;
}

void release(const Block& b)
{
    cudaFree(b.dev);
    cudaFreeHost(b.host);
}

}  // namespace

void pool_clear()
{
    std::vector<Block> all;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        all.swap(kept());
    }
    for (const Block& b : all) release(b);
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
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        std::vector<Block>& v = kept();
        size_t best = v.size();
        // the smallest that fits and wastes no more than a quarter (or 1 MB)
        for (size_t i = 0; i < v.size(); ++i)
            if (v[i].device == dev && v[i].bytes >= bytes && v[i].bytes - bytes <= bytes / 4 + ((size_t)1 << 20) &&
                (best == v.size() || v[i].bytes < v[best].bytes))
                best = i;
        if (best < v.size()) {
            *out = v[best];
            v.erase(v.begin() + (long)best);
            return cudaSuccess;
        }
    }
    Block b;
    b.bytes = bytes;
    b.device = dev;
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
    if (!idle) {
        release(b);
        return;
    }
    std::vector<Block> old;
    {
        std::lock_guard<std::mutex> lock(g_mutex);
        std::vector<Block>& v = kept();
        size_t total = b.bytes;
        for (const Block& k : v) total += k.bytes;
        if (b.bytes > kMostBytes) {
            old.push_back(b);
        } else {
            while (!v.empty() && (total > kMostBytes || v.size() >= kMostBlocks)) {
                total -= v.front().bytes;
                old.push_back(v.front());
                v.erase(v.begin());
            }
            v.push_back(b);
        }
    }
    for (const Block& k : old) release(k);
}

}  // namespace rr

extern "C" rr_status rr_release_cached(void)
{
    rr::pool_clear();
    return RR_OK;
}
