// Device memory for the library's buffers: cudaMalloc behind a small cache of
// freed blocks keyed by (device, exact size).
//
// A problem of a given shape allocates the same set of buffers every time (the
// factors alone are 8 (s/2+1) m_p^2 bytes), and cudaMalloc / cudaFree of
// gigabyte buffers cost milliseconds each, with cudaFree synchronising the
// device.  Repeated create / solve / destroy cycles (the end-to-end use of the
// API) therefore reuse the blocks of the previous problem.  The cache holds at
// most DEVMEM_CACHE_LIMIT bytes (oldest blocks are released first) and is
// emptied for the device when cudaMalloc runs out of memory, and entirely by
// fde_release_cached_memory().
//
// dev_free() callers guarantee that no queued GPU work still uses the block
// (every call site synchronises the problem's streams first); the block may be
// handed to another problem, on another stream, by the next dev_alloc().
#include <deque>
#include <mutex>
#include <unordered_map>
#include <vector>

#include "fde_internal.h"

namespace fde {

namespace {

constexpr size_t DEVMEM_CACHE_LIMIT = size_t(16) << 30;

struct Block {
    void* p;
    size_t bytes;
    int dev;
};

std::mutex g_mu;
std::deque<Block> g_cache;                     // freed blocks, oldest first
size_t g_cached = 0;                           // bytes held in g_cache
std::unordered_map<void*, Block> g_live;       // blocks handed out

constexpr size_t PINNED_CACHE_LIMIT = 16 << 20;  // bytes
constexpr size_t LU_CACHE_LIMIT = 8;
std::vector<void*> g_pinned[PINNED_CLASSES];   // returned pinned blocks by size
size_t g_pinned_cached = 0;                    // bytes held in g_pinned
std::unordered_map<void*, int> g_pinned_live;  // blocks handed out: their class
std::vector<LuStreams> g_lu;                   // returned LU streams

void release_cached(int dev) {  // g_mu held
    for (auto it = g_cache.begin(); it != g_cache.end();) {
        if (dev < 0 || it->dev == dev) {
            cudaFree(it->p);
            g_cached -= it->bytes;
            it = g_cache.erase(it);
        } else {
            ++it;
        }
    }
}

}  // namespace

int dev_alloc(void** p, size_t bytes) {
    *p = nullptr;
    if (bytes == 0) return FDE_OK;
    int dev = 0;
    FDE_CUDA_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(g_mu);
    for (auto it = g_cache.begin(); it != g_cache.end(); ++it) {
        if (it->dev == dev && it->bytes == bytes) {
            *p = it->p;
            g_cached -= bytes;
            g_live[*p] = *it;
            g_cache.erase(it);
            return FDE_OK;
        }
    }
    cudaError_t e = cudaMalloc(p, bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();  // clear, then retry with the cache of this device released
        release_cached(dev);
        e = cudaMalloc(p, bytes);
    }
    if (e != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        return set_error(FDE_ERR_ALLOC, std::string("cudaMalloc failed: ") + cudaGetErrorString(e));
    }
    g_live[*p] = Block{*p, bytes, dev};
    return FDE_OK;
}

void dev_free(void* p) {
    if (!p) return;
    std::lock_guard<std::mutex> lock(g_mu);
    auto it = g_live.find(p);
    if (it == g_live.end()) {  // not from dev_alloc
        cudaFree(p);
        return;
    }
    const Block b = it->second;
    g_live.erase(it);
    if (b.bytes > DEVMEM_CACHE_LIMIT) {
        cudaFree(p);
        return;
    }
    g_cache.push_back(b);
    g_cached += b.bytes;
    while (g_cached > DEVMEM_CACHE_LIMIT && !g_cache.empty()) {
        cudaFree(g_cache.front().p);
        g_cached -= g_cache.front().bytes;
        g_cache.pop_front();
    }
}

// A cache hit costs the problem that starts 150 us less than cudaMallocHost, and the one that
// ends 190 us less than cudaFreeHost, which waits for the device.
int pinned_alloc(size_t bytes, void** p) {
    const int c = pinned_class(bytes);
    if (c < PINNED_CLASSES) {
        bytes = PINNED_LEAST << c;
        std::lock_guard<std::mutex> lock(g_mu);
        if (!g_pinned[c].empty()) {
            *p = g_pinned[c].back();
            g_pinned[c].pop_back();
            g_pinned_cached -= bytes;
            g_pinned_live[*p] = c;
            return FDE_OK;
        }
    }
    *p = nullptr;
    const cudaError_t e = cudaHostAlloc(p, bytes, cudaHostAllocPortable);
    if (e != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        return set_error(FDE_ERR_ALLOC, std::string("cudaHostAlloc failed: ") + cudaGetErrorString(e));
    }
    std::lock_guard<std::mutex> lock(g_mu);
    g_pinned_live[*p] = c;
    return FDE_OK;
}

void pinned_free(void* p) {
    if (!p) return;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        const auto it = g_pinned_live.find(p);
        const int c = it->second;
        g_pinned_live.erase(it);
        if (c < PINNED_CLASSES && g_pinned_cached + (PINNED_LEAST << c) <= PINNED_CACHE_LIMIT) {
            g_pinned[c].push_back(p);
            g_pinned_cached += PINNED_LEAST << c;
            return;
        }
    }
    cudaFreeHost(p);
}

static void lu_streams_destroy(LuStreams& s) {
    for (cudaStream_t st : {s.hi, s.lo, s.x})
        if (st) cudaStreamDestroy(st);
    for (cudaEvent_t e : s.ev)
        if (e) cudaEventDestroy(e);
    s = LuStreams();
}

int lu_streams_take(LuStreams* s) {
    int dev = 0;
    FDE_CUDA_TRY(cudaGetDevice(&dev));
    {
        std::lock_guard<std::mutex> lock(g_mu);
        for (auto it = g_lu.begin(); it != g_lu.end(); ++it)
            if (it->dev == dev) {
                *s = *it;
                g_lu.erase(it);
                return FDE_OK;
            }
    }
    LuStreams n;
    int least = 0, greatest = 0;
    cudaError_t e = cudaDeviceGetStreamPriorityRange(&least, &greatest);
    if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&n.hi, cudaStreamNonBlocking, greatest);
    if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&n.lo, cudaStreamNonBlocking, least);
    // the cross tiles one level below the panel chain (the next diagonal kernel gets the SMs
    // first), above the interior updates
    const int mid = greatest < least ? greatest + 1 : greatest;
    if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&n.x, cudaStreamNonBlocking, mid);
    for (cudaEvent_t& ev : n.ev)
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e != cudaSuccess) {
        lu_streams_destroy(n);
        return cuda_error(e, "streams of the block LU");
    }
    n.dev = dev;
    *s = n;
    return FDE_OK;
}

void lu_streams_return(LuStreams* s) {
    if (!s->hi) return;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (g_lu.size() < LU_CACHE_LIMIT) {
            g_lu.push_back(*s);
            *s = LuStreams();
            return;
        }
    }
    lu_streams_destroy(*s);
}

int allow_smem(const void* kern, size_t bytes) {
    static std::mutex mu;
    static std::unordered_map<const void*, std::vector<size_t>> most;  // per kernel and device
    int dev = 0;
    FDE_CUDA_TRY(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lock(mu);
    std::vector<size_t>& m = most[kern];
    if ((int)m.size() <= dev) m.resize(dev + 1, 0);
    if (m[dev] >= bytes) return FDE_OK;
    FDE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    m[dev] = bytes;
    return FDE_OK;
}

int dev_release_cached() {
    std::lock_guard<std::mutex> lock(g_mu);
    cudaError_t first = cudaSuccess;
    for (std::vector<void*>& blocks : g_pinned) {
        for (void* p : blocks) {
            const cudaError_t e = cudaFreeHost(p);
            if (e != cudaSuccess && first == cudaSuccess) first = e;
        }
        blocks.clear();
    }
    g_pinned_cached = 0;
    for (LuStreams& l : g_lu) lu_streams_destroy(l);
    g_lu.clear();
    for (const Block& b : g_cache) {
        const cudaError_t e = cudaFree(b.p);
        if (e != cudaSuccess && first == cudaSuccess) first = e;
    }
    g_cache.clear();
    g_cached = 0;
    if (first != cudaSuccess) {
        cudaGetLastError();
        return set_error(FDE_ERR_CUDA, std::string("cudaFree failed: ") + cudaGetErrorString(first));
    }
    return FDE_OK;
}

}  // namespace fde
