// memory.cu against a fake CUDA runtime: one scenario a run (argv[1]), exit
// status 0 if it holds.  The fakes count, fail or block the calls they stand for.
#include <cuda.h>
#include <cuda_runtime.h>

#include <condition_variable>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <thread>

#include "memory.cuh"

namespace {
std::mutex g_mu;
std::condition_variable g_cv;
bool g_hold = false;          // cudaDeviceSynchronize and cudaFree block while set
int g_held = 0;               // calls blocked

void hold_point() {
    std::unique_lock<std::mutex> lk(g_mu);
    ++g_held;
    g_cv.notify_all();
    g_cv.wait(lk, [] { return !g_hold; });
    --g_held;
}

std::set<void *> g_live;      // blocks of cudaMalloc not yet freed
size_t g_next = 1 << 20;      // the next address
int g_waits = 0, g_mallocs = 0;
cudaError_t g_wait_status = cudaSuccess;
unsigned long long g_context = 1;  // the current context's id
std::set<size_t> g_pools_used;     // pools temporaries came from
size_t g_pools = 0, g_trims = 0;

CUresult current(CUcontext *c) {
    *c = reinterpret_cast<CUcontext>(0x100);
    return CUDA_SUCCESS;
}
CUresult context_id(CUcontext, unsigned long long *id) {
    *id = g_context;
    return CUDA_SUCCESS;
}

#define CHECK(c)                                               \
    do {                                                       \
        if (!(c)) {                                            \
            std::printf("line %d: %s\n", __LINE__, #c);        \
            return 1;                                          \
        }                                                      \
    } while (0)

void *get(size_t bytes) {
    void *p = nullptr;
    return spmv::dev_malloc(&p, bytes) == cudaSuccess ? p : nullptr;
}
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) {
    std::lock_guard<std::mutex> lk(g_mu);
    ++g_mallocs;
    *p = reinterpret_cast<void *>(g_next);
    g_next += (n + 255) / 256 * 256;
    g_live.insert(*p);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (!p) return cudaSuccess;
    hold_point();
    std::lock_guard<std::mutex> lk(g_mu);
    return g_live.erase(p) ? cudaSuccess : cudaErrorInvalidValue;
}
cudaError_t cudaDeviceSynchronize(void) {
    hold_point();
    ++g_waits;
    return g_wait_status;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) {
    *p = reinterpret_cast<cudaMemPool_t>(++g_pools);
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t keep) {
    g_trims += keep == 0;
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void **p, size_t, cudaMemPool_t pool, cudaStream_t) {
    g_pools_used.insert(reinterpret_cast<size_t>(pool));
    *p = &g_pools_used;
    return cudaSuccess;
}
cudaError_t cudaMallocAsync(void **, size_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *name, void **fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *found) {
    *fn = !std::strcmp(name, "cuCtxGetId") ? reinterpret_cast<void *>(&context_id) : reinterpret_cast<void *>(&current);
    *found = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
}

// a freed block is handed out again after a wait that succeeded, not before
static int reuse() {
    void *a = get(5000), *b = get(5000);
    CHECK(a && b && a != b);
    spmv::dev_free(a);
    CHECK(g_waits == 0);
    void *c = get(5000);  // of a's size: the library waits first
    CHECK(g_waits == 1 && c == a);
    spmv::dev_free(b);
    spmv::dev_settle();
    CHECK(g_waits == 2);
    CHECK(get(5000) == b && g_waits == 2 && g_mallocs == 2);
    return 0;
}

// where the wait fails (a stream of another thread is being captured, the
// context is broken) no freed block is handed out
static int failed_wait() {
    void *a = get(5000);
    spmv::dev_free(a);
    g_wait_status = cudaErrorStreamCaptureUnsupported;
    spmv::dev_settle();
    void *b = get(5000);
    CHECK(b && b != a && g_live.count(a));
    g_wait_status = cudaSuccess;
    CHECK(get(5000) == a);
    return 0;
}

// at most 64 MiB are kept, blocks over 8 MiB not at all
static int bounded() {
    void *big = get((8 << 20) + 1);
    spmv::dev_free(big);
    CHECK(!g_live.count(big));
    std::set<void *> blocks;
    for (int i = 0; i < 40; ++i) blocks.insert(get(4 << 20));
    CHECK(blocks.size() == 40);
    for (void *p : blocks) spmv::dev_free(p);
    CHECK(g_live.size() == 16);
    return 0;
}

// a thread that waits for the device, or frees a large block, holds up nobody else
static int threads() {
    void *a = get(5000), *big = get(size_t(9) << 20), *b = get(700);
    for (int round = 0; round < 2; ++round) {
        g_hold = true;
        std::thread t(round == 0 ? [](void *small, void *) { spmv::dev_free(small), spmv::dev_settle(); }
                                 : [](void *, void *large) { spmv::dev_free(large); },
                      a, big);
        {
            std::unique_lock<std::mutex> lk(g_mu);
            g_cv.wait(lk, [] { return g_held == 1; });
        }
        void *c = get(9000 << round);  // (blocks for good where the lock is held: the run is then ended from outside)
        CHECK(c && c != a);
        spmv::dev_free(c);
        if (round == 0) spmv::dev_free(b);  // freed after the wait began: not ready when it ends
        {
            std::lock_guard<std::mutex> lk(g_mu);
            g_hold = false;
        }
        g_cv.notify_all();
        t.join();
    }
    const int waits = g_waits;
    CHECK(get(5000) == a && g_waits == waits);
    CHECK(get(700) == b && g_waits == waits + 1);
    return 0;
}

// a device reset ends the context: nothing of it is handed out, used or listed
// again, nor freed, since its addresses are given anew
static int reset() {
    void *a = get(5000), *b = get(6000), *c = get(7000), *big = get(size_t(9) << 20), *t = nullptr;
    spmv::dev_free(a);
    spmv::dev_settle();
    spmv::dev_free(b);
    CHECK(spmv::dev_malloc_async(&t, 100, nullptr) == cudaSuccess);
    g_context = 2;
    const std::set<void *> others = g_live;  // somebody else's blocks in the new context
    CHECK(get(5000) != a && get(6000) != b && g_mallocs == 6);
    spmv::dev_free(c);  // of the old context
    spmv::dev_free(big);
    for (void *p : others) CHECK(g_live.count(p));
    CHECK(get(7000) != c);
    spmv::dev_settle();
    CHECK(get(7000) != c);
    CHECK(spmv::dev_malloc_async(&t, 100, nullptr) == cudaSuccess);
    CHECK(g_pools == 2 && g_pools_used == (std::set<size_t>{1, 2}));
    void *d = get(5000);  // the new one keeps its own
    spmv::dev_free(d);
    spmv::dev_settle();
    CHECK(get(5000) == d);
    return 0;
}

// everything kept can be given back
static int trim() {
    void *a = get(5000), *b = get(6000), *c = get(7000), *t = nullptr;
    CHECK(spmv::dev_malloc_async(&t, 100, nullptr) == cudaSuccess);
    spmv::dev_free(a);
    spmv::dev_settle();
    spmv::dev_free(b);
    g_wait_status = cudaErrorStreamCaptureUnsupported;
    CHECK(spmv::dev_trim() != cudaSuccess && g_live.size() == 3);
    g_wait_status = cudaSuccess;
    CHECK(spmv::dev_trim() == cudaSuccess);
    CHECK(g_live == std::set<void *>{c} && g_trims == 1);
    spmv::dev_free(c);
    CHECK(spmv::dev_trim() == cudaSuccess && g_live.empty());
    return 0;
}

int main(int argc, char **argv) {
    const std::map<std::string, int (*)()> all = {{"reuse", reuse}, {"failed_wait", failed_wait}, {"bounded", bounded},
                                                       {"threads", threads},   {"reset", reset},
                                                       {"trim", trim}};
    const auto it = all.find(argc > 1 ? argv[1] : "");
    return it == all.end() ? 2 : it->second();
}
