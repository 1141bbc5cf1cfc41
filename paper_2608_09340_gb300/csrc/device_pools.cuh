// The memory pools of the library, host code only.
#pragma once

#include <cuda_runtime_api.h>
#include <stddef.h>

#include <mutex>

namespace krl {

// Device memory comes from two stream-ordered pools of the library's own per
// device, one for what grids and batches keep, one for the scratch of a call,
// so that creating, replacing and destroying lines, and calls that the caller
// waits for, do not map and unmap memory each time: a synchronisation unmaps
// what a pool holds unused above its threshold, with the default pool all of
// it (7 ms of a 27 ms ray trace with 4.3 GB of scratch). The thresholds bound
// what stays mapped; with the device's last grid the scratch pool is emptied.
struct DevicePools {
    cudaMemPool_t kept = nullptr, scratch = nullptr;
    int grids = 0;
};
constexpr unsigned long long kKeptIdle = 256ull << 20, kScratchIdle = 6ull << 30;
constexpr int kMaxDevices = 64;
inline std::mutex g_pool_mu;
inline DevicePools g_pools[kMaxDevices];

inline cudaError_t make_pool(int dev, unsigned long long idle, cudaMemPool_t* out)
{
    cudaMemPoolProps p{};
    p.allocType = cudaMemAllocationTypePinned;
    p.location.type = cudaMemLocationTypeDevice;
    p.location.id = dev;
    cudaError_t e = cudaMemPoolCreate(out, &p);
    if (e == cudaSuccess) e = cudaMemPoolSetAttribute(*out, cudaMemPoolAttrReleaseThreshold, &idle);
    return e;
}

// The current device's pools, made on first use. grids: change of its count
// of grids.
inline cudaError_t device_pools(DevicePools* out, int grids = 0)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_pool_mu);
    DevicePools& P = g_pools[dev];
    if (!P.kept) e = make_pool(dev, kKeptIdle, &P.kept);
    if (e == cudaSuccess && !P.scratch) e = make_pool(dev, kScratchIdle, &P.scratch);
    P.grids += grids;
    *out = P;
    return e;
}

// From one of the pools, in the order of s. When there is no memory, once more
// after unmapping what both hold unused. For kept memory, whose calls wait for
// s anyway, that includes what is being freed behind work in flight on other
// streams (scratch of several GB behind a ray trace): such blocks can be
// unmapped only when that work has ended, so the device is waited for. Scratch
// stays in stream order: its calls have a way without it.
inline cudaError_t pool_alloc(void** p, size_t bytes, bool scratch, cudaStream_t s)
{
    DevicePools P;
    cudaError_t e = device_pools(&P);
    if (e != cudaSuccess) return e;
    const cudaMemPool_t pool = scratch ? P.scratch : P.kept;
    e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    if (e == cudaErrorMemoryAllocation) {
        (void)cudaGetLastError();
        cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
        if (!scratch && cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone &&
            cudaDeviceSynchronize() != cudaSuccess)
            (void)cudaGetLastError();
        (void)cudaMemPoolTrimTo(P.kept, 0);
        (void)cudaMemPoolTrimTo(P.scratch, 0);
        e = cudaMallocFromPoolAsync(p, bytes, pool, s);
    }
    return e;
}

// Unmaps what the current device's pools hold unused, what is being freed
// behind work in flight included.
inline cudaError_t pools_trim()
{
    DevicePools P;
    cudaError_t e = device_pools(&P);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemPoolTrimTo(P.kept, 0);
    if (e == cudaSuccess) e = cudaMemPoolTrimTo(P.scratch, 0);
    return e;
}

}  // namespace krl
