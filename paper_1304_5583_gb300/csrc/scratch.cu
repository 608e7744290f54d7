// Stream-ordered scratch of the entry points that are called without a
// workspace.  The device's default pool returns its memory to the system at
// every synchronisation, and every entry point synchronises, so each call mapped
// its scratch anew: 190 us of a 285 us lrr_gemm_f32 call.  The library's own pool
// keeps up to kKeep bytes per device between calls (what is above goes back at
// the next synchronisation) and is destroyed with the library.
#include <mutex>

#include "common.cuh"
#include "kernels.cuh"

namespace lrr {
namespace {

constexpr uint64_t kKeep = uint64_t(64) << 20;

struct Pools {
    std::mutex mu;
    cudaMemPool_t pool[64] = {};
    ~Pools() {
        for (auto p : pool)
            if (p) (void)cudaMemPoolDestroy(p);     // fails harmlessly after the runtime has gone
    }
};
Pools g_pools;

// the current device's pool (nullptr: the default pool is used instead)
cudaMemPool_t device_pool() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lock(g_pools.mu);
    if (!g_pools.pool[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        uint64_t keep = kKeep;
        if (cudaMemPoolCreate(&p, &props) != cudaSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) (void)cudaGetLastError();
        g_pools.pool[dev] = p;
    }
    return g_pools.pool[dev];
}

}  // namespace

cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t s) {
    cudaMemPool_t pool = device_pool();
    return pool ? cudaMallocFromPoolAsync(p, bytes, pool, s) : cudaMallocAsync(p, bytes, s);
}

}  // namespace lrr
