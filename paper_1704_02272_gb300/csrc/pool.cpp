// Scratch memory of the calls that allocate it themselves (pfac_match,
// pfac_verify): a stream-ordered pool of the library's own per context that
// keeps up to POOL_KEEP bytes between calls.  The device's default pool gives
// everything back whenever the stream is waited for, so that every call mapped
// its workspace again (a call on 1 MiB of text: 0.32 ms alone).
#include <cuda_runtime.h>

#include <mutex>

#include "internal.h"

namespace pfac {

namespace {

constexpr int MAX_DEV = 64;
constexpr int MAX_CTX = 8;  // contexts of a device that get a pool
constexpr uint64_t POOL_KEEP = 64ull << 20;

// A pool and the context it was made in, by the context's id: a context that
// takes another's place (cudaDeviceReset) may lie at the same address.  Pools
// of contexts that are gone stay listed, unused: their handles cannot be told
// from live ones to destroy them.
struct Pool {
    uint64_t ctx = 0;
    cudaMemPool_t pool = nullptr;
};
std::mutex g_mu;
Pool g_pool[MAX_DEV][MAX_CTX];

// This context's pool, made on the first call with `make`; nullptr when there
// is none or none can be had (the default pool serves).
cudaMemPool_t context_pool(bool make) {
    int dev = 0;
    const uint64_t ctx = current_context_id();
    if (!ctx || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEV) return nullptr;
    std::lock_guard<std::mutex> lk(g_mu);
    Pool *p = g_pool[dev], *end = p + MAX_CTX;
    while (p < end && p->pool && p->ctx != ctx) p++;
    if (p == end) return nullptr;
    if (p->pool || !make) return p->pool;
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
    p->ctx = ctx;
    p->pool = pool;
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
        const cudaMemPool_t pool = context_pool(true);
        if (pool) {
            const cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, st);
            if (e == cudaSuccess) return e;
            cudaGetLastError();
        }
    }
    return cudaMallocAsync(p, bytes, st);
}

void scratch_trim() {
    const cudaMemPool_t pool = context_pool(false);
    if (!pool) return;
    // frees still pending on a stream are not the pool's to give back yet
    if (cudaDeviceSynchronize() != cudaSuccess || cudaMemPoolTrimTo(pool, 0) != cudaSuccess) cudaGetLastError();
}

}  // namespace pfac
