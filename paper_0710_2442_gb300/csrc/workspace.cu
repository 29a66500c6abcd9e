// workspace.cu -- the library's memory pools: one per device and use, with
// stream-ordered allocation, bounded in what they keep, and given back on request.
#include "internal.h"

namespace wl {

namespace {

std::mutex g_pools_mutex;
cudaMemPool_t g_pools[kPools][64] = {};

int current_device() {
    int dev = 0;
    WL_CUDA(cudaGetDevice(&dev));
    WL_REQUIRE(dev >= 0 && dev < 64, "device ordinal out of range");
    return dev;
}

cudaMemPool_t pool_of(Pool which) {
    const int dev = current_device();
    std::lock_guard<std::mutex> lk(g_pools_mutex);
    cudaMemPool_t& pool = g_pools[which][dev];
    if (!pool) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        WL_CUDA(cudaMemPoolCreate(&p, &props));
        unsigned long long keep = ~0ULL;
        if (which != POOL_STATELESS) {
            size_t free_bytes = 0, total = 0;
            WL_CUDA(cudaMemGetInfo(&free_bytes, &total));
            keep = total / 32;
        }
        WL_CUDA(cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep));
        pool = p;
    }
    return pool;
}

thread_local bool t_active = false;
thread_local cudaStream_t t_stream = nullptr;

}  // namespace

cudaError_t pool_alloc(void** p, size_t n, Pool which, cudaStream_t st) {
    cudaError_t e = cudaMallocFromPoolAsync(p, n, pool_of(which), st);
    if (e == cudaErrorMemoryAllocation) {  // what the others keep
        (void)cudaGetLastError();
        trim_pools();
        e = cudaMallocFromPoolAsync(p, n, pool_of(which), st);
    }
    return e;
}

void trim_pools() {
    const int dev = current_device();
    std::lock_guard<std::mutex> lk(g_pools_mutex);
    for (int k = 0; k < kPools; k++)
        if (g_pools[k][dev]) WL_CUDA(cudaMemPoolTrimTo(g_pools[k][dev], 0));
}

cudaError_t device_alloc(void** p, size_t n) {
    cudaError_t e = cudaMalloc(p, n);
    if (e == cudaErrorMemoryAllocation) {
        (void)cudaGetLastError();
        trim_pools();
        e = cudaMalloc(p, n);
    }
    return e;
}

WorkspaceScope::WorkspaceScope(cudaStream_t st) : before_(t_active), st_before_(t_stream) {
    t_active = true;
    t_stream = st;
}
WorkspaceScope::~WorkspaceScope() {
    t_active = before_;
    t_stream = st_before_;
}

void* workspace_alloc(size_t n, cudaStream_t* st) {
    if (!t_active) return nullptr;
    void* p = nullptr;
    WL_CUDA(pool_alloc(&p, n, POOL_SOLVE, t_stream));
    *st = t_stream;
    return p;
}

}  // namespace wl
