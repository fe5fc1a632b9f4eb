// pool.cpp -- the workspace's memory pool.
//
// A call allocates its workspace stream-ordered and frees it before it
// returns.  From the device's default pool every freed byte went back to the
// system at the call's last synchronisation, and the next call mapped it anew:
// about 2.7 ms for each GB (GB300: 11 of the 22 ms of one emulated FP64 step at
// n = 8192, 4 of the 7.5 ms of a low-precision one).  The library keeps one
// pool of its own per context that holds on to at most kPoolKeep bytes between
// calls.  The driver takes unused bytes back from it when any allocation of the
// process would otherwise fail (measured: cudaMalloc of 3 GB more than was
// free, with 6.4 GB held, succeeds and leaves the pool empty), and a call that
// used more gives the excess back as before.
//
// The pool is the driver's: it is safe with several threads, and memory freed
// on one stream and reused on another is ordered by the driver.  A pool
// belongs to a context and goes with it: each context has its own, found by the
// context's id, which no later context gets (after cudaDeviceReset a device has
// a new one).
#include <cuda.h>
#include <cuda_runtime.h>

#include <mutex>

#include "internal.h"

namespace jac {

namespace {

constexpr unsigned long long kPoolKeep = 8ull << 30;   // 3 % of the device's memory
constexpr int kPoolContexts = 64;   // looked after at once; beyond them the first one's entry is used anew

struct Entry {
    unsigned long long ctx = 0;
    cudaMemPool_t pool = nullptr;
};

std::mutex g_mu;
Entry g_pool[kPoolContexts];
int g_next = 0;

using CtxGetId = CUresult (*)(CUcontext, unsigned long long*);

// The pool of the current device's context, or null (no driver, no context).
cudaMemPool_t pool_here()
{
    static const CtxGetId ctx_id = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return (CtxGetId)f;
    }();
    int dev = -1;
    unsigned long long id = 0;
    // (a thread without a context gets the device's primary one; cudaFree(nullptr)
    // would do that too, but is refused while any thread captures a graph)
    if (!ctx_id || cudaGetDevice(&dev) != cudaSuccess ||
        (ctx_id(nullptr, &id) != CUDA_SUCCESS && (cudaSetDevice(dev) != cudaSuccess || ctx_id(nullptr, &id) != CUDA_SUCCESS))) {
        cudaGetLastError();
        return nullptr;
    }
    std::lock_guard<std::mutex> lock(g_mu);
    for (const Entry& e : g_pool)
        if (e.pool && e.ctx == id) return e.pool;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    unsigned long long keep = kPoolKeep;
    if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        cudaMemPoolDestroy(p);
        return nullptr;
    }
    g_pool[g_next] = Entry{id, p};
    g_next = (g_next + 1) % kPoolContexts;
    return p;
}

}  // namespace

cudaError_t workspace_alloc(void** p, size_t bytes, cudaStream_t s)
{
    if (cudaMemPool_t pool = pool_here()) {
        if (cudaMallocFromPoolAsync(p, bytes, pool, s) == cudaSuccess) return cudaSuccess;
        cudaGetLastError();
    }
    return cudaMallocAsync(p, bytes, s);
}

}  // namespace jac
