// Scratch memory of the calls that allocate it themselves (pfac_match,
// pfac_verify): a stream-ordered pool of the library's own per device that
// keeps up to POOL_KEEP bytes between calls.  The device's default pool gives
// everything back whenever the stream is waited for, so that every call mapped
// its workspace again (a call on 1 MiB of text: 0.32 ms alone).
#include <cuda_runtime.h>

#include <mutex>

#include "internal.h"

namespace pfac {

namespace {

constexpr int MAX_DEV = 64;
constexpr uint64_t POOL_KEEP = 64ull << 20;

// A device's pool and the context it was made in: after the context is
// replaced (cudaDeviceReset) another one is made.
struct Pool {
    void *ctx = nullptr;
    cudaMemPool_t pool = nullptr;
};
std::mutex g_mu;
Pool g_pool[MAX_DEV];

// This device's pool, or nullptr (no pool can be had: the default one serves).
cudaMemPool_t device_pool() {
    int dev = 0;
    void *ctx = current_context();
    if (!ctx || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEV) return nullptr;
    std::lock_guard<std::mutex> lk(g_mu);
    Pool &p = g_pool[dev];
    if (p.pool && p.ctx == ctx) return p.pool;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    uint64_t keep = POOL_KEEP;
    if (cudaMemPoolCreate(&pool, &props) != cudaSuccess ||
        cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
        cudaGetLastError();
        if (pool) cudaMemPoolDestroy(pool);
        return nullptr;
    }
    p.ctx = ctx;
    p.pool = pool;
    return pool;
}

}  // namespace

cudaError_t scratch_alloc(void **p, size_t bytes, cudaStream_t st) {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(st, &cap) != cudaSuccess) {
        cudaGetLastError();
        cap = cudaStreamCaptureStatusActive;
    }
    if (cap == cudaStreamCaptureStatusNone) {
        const cudaMemPool_t pool = device_pool();
        if (pool) {
            const cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, st);
            if (e == cudaSuccess) return e;
            cudaGetLastError();
        }
    }
    return cudaMallocAsync(p, bytes, st);
}

void scratch_trim() {
    const cudaMemPool_t pool = device_pool();
    if (pool && cudaMemPoolTrimTo(pool, 0) != cudaSuccess) cudaGetLastError();
}

}  // namespace pfac
