// Device memory of the library's objects and temporaries, from one
// stream-ordered pool per device.
//
// cudaMalloc and cudaFree take 10 to 200 us each and synchronise the device,
// and the default pool gives its memory back at every synchronisation, so an
// encode of a 22M-nonzero matrix (18 allocations, one synchronisation in the
// middle) spent about 1 ms of its 1.4 ms in the allocator. The library's pool
// keeps up to kKeep bytes of freed memory for the next call and returns the
// rest to the system at the next synchronisation; when an allocation fails,
// and when the user asks for it (packsell_trim), everything unused goes back.
#include <cuda_runtime.h>

#include <mutex>

#include "internal.h"

namespace packsell {
namespace {

constexpr int kMaxDevices = 64;
constexpr unsigned long long kKeep = 2ull << 30;  // freed bytes kept per device at most

std::mutex g_mu;
cudaMemPool_t g_pool[kMaxDevices] = {};

cudaError_t pool_of(int dev, cudaMemPool_t *out) {
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_pool[dev]) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        const cudaError_t e = cudaMemPoolCreate(&g_pool[dev], &props);
        if (e != cudaSuccess) return e;
    }
    *out = g_pool[dev];
    return cudaSuccess;
}

// What the pool may hold is what is in use plus kKeep: the threshold counts
// the live memory too, so it moves with it.
void set_threshold(cudaMemPool_t pool) {
    unsigned long long used = 0;
    if (cudaMemPoolGetAttribute(pool, cudaMemPoolAttrUsedMemCurrent, &used) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    used += kKeep;
    if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &used) != cudaSuccess)
        cudaGetLastError();
}

}  // namespace

cudaError_t pool_get(void **p, size_t bytes, cudaStream_t s) {
    *p = nullptr;
    int dev = 0;
    cudaMemPool_t pool;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = pool_of(dev, &pool);
    if (e != cudaSuccess) return e;
    bytes = bytes ? bytes : 16;
    e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    if (e == cudaErrorMemoryAllocation) {
        // what is freed on any stream counts; a stream under capture must not be
        // synchronised with
        cudaGetLastError();
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
            flush_destroyed(dev);
            cudaDeviceSynchronize();
        }
        cudaGetLastError();
        cudaMemPoolTrimTo(pool, 0);
        e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    }
    if (e == cudaSuccess) set_threshold(pool);
    return e;
}

cudaError_t pool_trim() {
    int dev = 0;
    cudaMemPool_t pool;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) {
        flush_destroyed(dev);
        e = cudaDeviceSynchronize();
    }
    if (e == cudaSuccess) e = pool_of(dev, &pool);
    if (e == cudaSuccess) e = cudaMemPoolTrimTo(pool, 0);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

void pool_put(void *p, cudaStream_t s) {
    if (!p) return;
    int dev = 0;
    cudaMemPool_t pool;
    if (cudaFreeAsync(p, s) != cudaSuccess) {
        // cudaFree of pool memory waits for nothing: only after the device has
        // finished, or not at all
        cudaGetLastError();
        if (cudaDeviceSynchronize() == cudaSuccess) cudaFree(p);
        cudaGetLastError();
    }
    if (cudaGetDevice(&dev) == cudaSuccess && pool_of(dev, &pool) == cudaSuccess) set_threshold(pool);
}

}  // namespace packsell
