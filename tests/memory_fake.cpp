// memory.cu against a fake CUDA runtime: one scenario a run (argv[1]), exit
// status 0 if it holds.  The fakes count, fail or block the calls they stand for.
#include <cuda_runtime.h>

#include <condition_variable>
#include <cstdio>
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
cudaError_t cudaMemPoolCreate(cudaMemPool_t *, const cudaMemPoolProps *) { return cudaErrorNotSupported; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **, size_t, cudaMemPool_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaMallocAsync(void **, size_t, cudaStream_t) { return cudaErrorNotSupported; }
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

int main(int argc, char **argv) {
    const std::map<std::string, int (*)()> all = {{"reuse", reuse}, {"failed_wait", failed_wait}, {"bounded", bounded},
                                                       {"threads", threads}};
    const auto it = all.find(argc > 1 ? argv[1] : "");
    return it == all.end() ? 2 : it->second();
}
