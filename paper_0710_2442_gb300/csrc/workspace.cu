// workspace.cu -- the solves' workspace: a memory pool per device with
// stream-ordered allocation (WorkspaceScope in internal.h).
#include "internal.h"

namespace wl {

namespace {

thread_local bool t_active = false;
thread_local cudaStream_t t_stream = nullptr;

cudaMemPool_t solve_pool() {
    static std::mutex m;
    static cudaMemPool_t pools[64] = {};
    int dev = 0;
    WL_CUDA(cudaGetDevice(&dev));
    WL_REQUIRE(dev >= 0 && dev < 64, "device ordinal out of range");
    std::lock_guard<std::mutex> lk(m);
    if (!pools[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool = nullptr;
        WL_CUDA(cudaMemPoolCreate(&pool, &props));
        size_t free_bytes = 0, total = 0;
        WL_CUDA(cudaMemGetInfo(&free_bytes, &total));
        unsigned long long keep = total / 32;
        WL_CUDA(cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep));
        pools[dev] = pool;
    }
    return pools[dev];
}

}  // namespace

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
    WL_CUDA(cudaMallocFromPoolAsync(&p, n, solve_pool(), t_stream));
    *st = t_stream;
    return p;
}

}  // namespace wl
