// Device memory (memory.cuh).
//
// A cudaMalloc and cudaFree pair costs 70 us and more, and a handle holds up
// to twenty small arrays (work items, join scratch, row pointers of small
// matrices), so blocks of up to SMALL_MOST bytes are kept: a freed block waits
// until the library has waited for the device (work launched before the free
// may still use it) and is then handed out again.  Where that wait fails, the
// blocks go on waiting.  Temporaries of one call come from a stream-ordered
// pool of the library that keeps POOL_KEEP bytes mapped across the call's own
// synchronisations (the default pool unmaps at each: 2 us per MB to map and
// unmap).  At most SMALL_KEEP + POOL_KEEP bytes are kept per device (0.1% of
// it); what exceeds them goes back at once, the rest when an allocation fails or
// the caller asks for it (spmv_trim).
//
// Blocks and pool belong to a context, not to a device: cudaDeviceReset ends
// the context and with it everything kept, and a context of the driver API has
// memory of its own.  The tables go by the id of the context, which the driver
// never gives twice; what belonged to a context that has ended is not touched
// again, not even freed (its addresses may be someone else's by then).
#include "memory.cuh"

#include <cuda.h>

#include <cstdint>
#include <cstdlib>
#include <map>
#include <mutex>
#include <new>
#include <unordered_map>
#include <utility>
#include <vector>

namespace spmv {

namespace {

thread_local long long g_alloc_count = 0;

// read on every allocation so a test can set and clear it at will
bool fault_injected() {
    const char *v = std::getenv("SPMV_FAULT_ALLOC");
    ++g_alloc_count;
    if (!v || !*v) return false;
    const long long k = std::atoll(v);
    return k > 0 && g_alloc_count == k;
}

constexpr size_t SMALL_MOST = size_t(8) << 20, SMALL_KEEP = size_t(64) << 20, POOL_KEEP = size_t(256) << 20;

struct Context {
    CUcontext handle = nullptr;
    uint64_t id = 0;  // 0: none to be had; nothing is kept then
};
struct Block {
    size_t size;  // 0: larger than SMALL_MOST, not kept
    Context ctx;
};
// what is kept of one context
struct Kept {
    std::map<size_t, std::vector<void *>> ready;      // idle blocks by size
    std::vector<std::pair<size_t, void *>> waiting;   // freed since the device was last waited for
    size_t bytes = 0;                                 // in the two
    cudaMemPool_t pool = nullptr;
    bool pool_tried = false;
};
std::mutex g_mem_mu;  // guards the tables; not held while the device is waited for or memory mapped
std::unordered_map<void *, Block> g_blocks;  // every block handed out or kept
std::map<uint64_t, Kept> g_kept;             // by context

template <typename F>
F driver(const char *name) {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    if (cudaGetDriverEntryPointByVersion(name, &fn, 12000, cudaEnableDefault, &found) != cudaSuccess ||
        found != cudaDriverEntryPointSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    return reinterpret_cast<F>(fn);
}

// id of a context; 0 if it has ended
uint64_t id_of(CUcontext handle) {
    static const auto get = driver<CUresult (*)(CUcontext, unsigned long long *)>("cuCtxGetId");
    unsigned long long id = 0;
    return get && handle && get(handle, &id) == CUDA_SUCCESS ? id : 0;
}

Context current_context() {
    static const auto get = driver<CUresult (*)(CUcontext *)>("cuCtxGetCurrent");
    Context c;
    if (cudaFree(nullptr) != cudaSuccess) cudaGetLastError();  // (makes the device's context if there is none)
    else if (get && get(&c.handle) == CUDA_SUCCESS) c.id = id_of(c.handle);
    return c;
}

// four sizes an octave: at most a quarter more than asked for
size_t block_size(size_t bytes) {
    size_t s = 256;
    while (s < bytes) s *= 2;
    if (s <= 256) return s;
    const size_t quarter = s / 8;
    size_t t = s / 2;
    while (t < bytes) t += quarter;
    return (t + 255) / 256 * 256;
}

// a failure leaves no error behind for the next launch's check
void free_now(void *p) {
    if (cudaFree(p) != cudaSuccess) cudaGetLastError();
}

// waits for the device, then makes the blocks freed before the wait ready
void settle(uint64_t ctx) {
    std::vector<std::pair<size_t, void *>> w;
    {
        std::lock_guard<std::mutex> lk(g_mem_mu);
        auto it = g_kept.find(ctx);
        if (it == g_kept.end() || it->second.waiting.empty()) return;
        w.swap(it->second.waiting);
    }
    const bool idle = cudaDeviceSynchronize() == cudaSuccess;
    if (!idle) cudaGetLastError();
    size_t left = 0;  // blocks the host has no memory to list: they go back
    {
        std::lock_guard<std::mutex> lk(g_mem_mu);
        Kept &k = g_kept.find(ctx)->second;
        for (const auto &b : w) try {
                if (idle) k.ready[b.first].push_back(b.second);
                else k.waiting.push_back(b);
            } catch (const std::bad_alloc &) {
                k.bytes -= b.first;
                g_blocks.erase(b.second);
                w[left++] = b;
            }
    }
    for (size_t i = 0; i < left; ++i) free_now(w[i].second);
}

// a ready block of the size, or null; *waits: blocks of the size are waiting
void *take(uint64_t ctx, size_t size, bool *waits) {
    *waits = false;
    std::lock_guard<std::mutex> lk(g_mem_mu);
    auto it = g_kept.find(ctx);
    if (it == g_kept.end()) return nullptr;
    Kept &k = it->second;
    auto r = k.ready.find(size);
    if (r != k.ready.end() && !r->second.empty()) {
        void *p = r->second.back();
        r->second.pop_back();
        k.bytes -= size;
        return p;
    }
    for (const auto &w : k.waiting) *waits = *waits || w.first == size;
    return nullptr;
}

// gives back everything kept of the current context (blocks that another thread is waiting for stay)
void give_back(uint64_t ctx) {
    std::map<size_t, std::vector<void *>> ready;
    std::vector<std::pair<size_t, void *>> waiting;
    cudaMemPool_t pool;
    {
        std::lock_guard<std::mutex> lk(g_mem_mu);
        auto it = g_kept.find(ctx);
        if (it == g_kept.end()) return;
        Kept &k = it->second;
        ready.swap(k.ready);
        waiting.swap(k.waiting);
        pool = k.pool;
        auto unlist = [&](size_t size, void *p) {
            k.bytes -= size;
            g_blocks.erase(p);
        };
        for (const auto &r : ready)
            for (void *p : r.second) unlist(r.first, p);
        for (const auto &w : waiting) unlist(w.first, w.second);
    }
    for (const auto &r : ready)
        for (void *p : r.second) free_now(p);
    for (const auto &w : waiting) free_now(w.second);
    if (pool) cudaMemPoolTrimTo(pool, 0);
}

// the library's pool of the current context; null where it cannot be made
cudaMemPool_t pool_of(uint64_t ctx) {
    int dev = 0;
    if (!ctx || cudaGetDevice(&dev) != cudaSuccess) return nullptr;
    std::lock_guard<std::mutex> lk(g_mem_mu);
    Kept &k = g_kept[ctx];
    if (k.pool_tried) return k.pool;
    k.pool_tried = true;
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    uint64_t keep = POOL_KEEP;
    if (cudaMemPoolCreate(&k.pool, &props) != cudaSuccess ||
        cudaMemPoolSetAttribute(k.pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        k.pool = nullptr;
    }
    return k.pool;
}

}  // namespace

void reset_alloc_count() { g_alloc_count = 0; }

cudaError_t dev_malloc(void **p, size_t bytes) {
    *p = nullptr;
    if (fault_injected()) return cudaErrorMemoryAllocation;
    const Context c = current_context();
    const uint64_t ctx = c.id;
    const size_t size = ctx && bytes <= SMALL_MOST ? block_size(bytes) : 0;
    if (size) {
        bool waits = false;
        *p = take(ctx, size, &waits);
        if (!*p && waits) {
            settle(ctx);
            *p = take(ctx, size, &waits);
        }
        if (*p) return cudaSuccess;
    }
    cudaError_t e = cudaMalloc(p, size ? size : bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        give_back(ctx);
        e = cudaMalloc(p, size ? size : bytes);
    }
    if (e != cudaSuccess) {
        *p = nullptr;
        return e;
    }
    if (ctx) try {
            std::lock_guard<std::mutex> lk(g_mem_mu);
            g_blocks[*p] = Block{size, c};
        } catch (const std::bad_alloc &) {  // unlisted: goes back at once when freed
        }
    return e;
}

void dev_free(void *p) {
    if (!p) return;
    const uint64_t ctx = current_context().id;
    {
        std::lock_guard<std::mutex> lk(g_mem_mu);
        auto it = g_blocks.find(p);
        if (it != g_blocks.end()) {
            const Block b = it->second;
            if (ctx != b.ctx.id && id_of(b.ctx.handle) != b.ctx.id) {
                g_blocks.erase(it);
                return;
            }
            if (b.size && ctx == b.ctx.id) try {
                Kept &k = g_kept[ctx];
                if (k.bytes + b.size <= SMALL_KEEP) {
                    k.waiting.emplace_back(b.size, p);
                    k.bytes += b.size;
                    return;
                }
            } catch (const std::bad_alloc &) {
            }
            g_blocks.erase(it);  // before the address can be given out anew
        }
    }
    free_now(p);
}

cudaError_t dev_trim() {
    const uint64_t ctx = current_context().id;
    const cudaError_t e = cudaDeviceSynchronize();
    if (e == cudaSuccess) give_back(ctx);
    return e;
}

void dev_settle() { settle(current_context().id); }

cudaError_t dev_malloc_async(void **p, size_t bytes, cudaStream_t s) try {
    *p = nullptr;
    if (fault_injected()) return cudaErrorMemoryAllocation;
    const uint64_t ctx = current_context().id;
    cudaMemPool_t pool = pool_of(ctx);
    if (!pool) return cudaMallocAsync(p, bytes, s);
    cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        give_back(ctx);
        e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    }
    return e;
} catch (const std::bad_alloc &) {
    return cudaErrorMemoryAllocation;
}

}  // namespace spmv
