// helm_mem.cu - device memory of a context: a stream-ordered pool that keeps what a call frees.
//
// The default pool gives everything back at each synchronisation, so every call mapped its
// workspace anew. Of a preconditioner call (786 us on the 1041 x 1041 grid with one right-hand side,
// some 350 us of kernels) half was allocation, copies of a few bytes and synchronisations; with the
// pool, one upload per call and one synchronisation it takes 389 us, a 320-right-hand-side solve
// (4 GB of workspace) 4 ms less.
#include <algorithm>
#include <atomic>
#include <vector>

#include "helm_internal.h"

namespace helm {

namespace {
std::mutex g_mu;
std::vector<std::pair<int, cudaMemPool_t>> g_pools;   // (device, pool) of every context
std::atomic<unsigned long long> g_allocs{0};
}  // namespace

void pool_create(helm_ctx* ctx) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = ctx->device;
    size_t fr = 0, total = 0;
    cudaMemPool_t pool = nullptr;
    if (cudaMemGetInfo(&fr, &total) != cudaSuccess || cudaMemPoolCreate(&pool, &props) != cudaSuccess) {
        cudaGetLastError();   // without a pool of its own the context uses the device's default one
        return;
    }
    uint64_t keep = total / 32;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    ctx->pool = pool;
    std::lock_guard<std::mutex> g(g_mu);
    g_pools.emplace_back(ctx->device, pool);
}

void pool_destroy(helm_ctx* ctx) {
    if (!ctx->pool) return;
    {
        std::lock_guard<std::mutex> g(g_mu);
        g_pools.erase(std::remove(g_pools.begin(), g_pools.end(), std::make_pair(ctx->device, ctx->pool)),
                      g_pools.end());
    }
    cudaMemPoolDestroy(ctx->pool);   // memory still in use (a model that outlives its context) is freed later
    ctx->pool = nullptr;
}

cudaError_t pool_alloc(helm_ctx* ctx, void** p, size_t bytes, cudaStream_t s) {
    g_allocs.fetch_add(1, std::memory_order_relaxed);
    auto get = [&] {
        return ctx->pool ? cudaMallocFromPoolAsync(p, bytes, ctx->pool, s) : cudaMallocAsync(p, bytes, s);
    };
    cudaError_t e = get();
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    {
        // what the contexts of this device hold unused goes back first
        std::lock_guard<std::mutex> g(g_mu);
        for (const auto& q : g_pools)
            if (q.first == ctx->device) cudaMemPoolTrimTo(q.second, 0);
    }
    return get();
}

size_t pool_unused(helm_ctx* ctx) {
    if (!ctx->pool) return 0;
    uint64_t held = 0, used = 0;
    if (cudaMemPoolGetAttribute(ctx->pool, cudaMemPoolAttrReservedMemCurrent, &held) != cudaSuccess ||
        cudaMemPoolGetAttribute(ctx->pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return held > used ? (size_t)(held - used) : 0;
}

}  // namespace helm

extern "C" uint64_t helm_alloc_count(void) { return (uint64_t)helm::g_allocs.load(std::memory_order_relaxed); }
