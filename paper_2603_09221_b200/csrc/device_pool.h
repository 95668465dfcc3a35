// Device memory of the handles' workspaces: one pool per device, shared by its handles, so that a program that makes handles
// for changing shapes does not pay a cudaMalloc (0.2 to 2 ms above 1 MB) for each.  Host code only.
//
// The pool keeps at most kPoolKeep bytes that no handle uses.  It lives as long as some handle of the device does: the
// last one to go destroys the pool and its stream.  Every function may be called from any thread; a buffer belongs to
// one handle, and between that handle's pool_enter and pool_leave the pool cannot go away.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <mutex>

namespace ttc {
namespace mem {

constexpr int kMaxPoolDevices = 64;
constexpr unsigned long long kPoolKeep = 256ull << 20;
constexpr size_t kPoolLargest = 64ull << 20;    // above, cudaMalloc: the pool maps gigabytes slower (21 against 13 ms)

struct DevicePool {
    std::mutex lock;                     // guards everything below
    cudaMemPool_t pool = nullptr;
    cudaStream_t stream = nullptr;       // orders allocations and releases; nothing else runs on it
    long long handles = 0;
};
inline DevicePool g_pools[kMaxPoolDevices];

struct DevBuf {
    void* ptr = nullptr;
    size_t bytes = 0;
    cudaStream_t stream = nullptr;       // the pool's stream, or null for memory from cudaMalloc
};

// (the device is current, here and below)  Where the pool cannot be made, buffers come from cudaMalloc until a later
// handle makes it; each buffer remembers where it came from.
inline void pool_enter(int device)
{
    if (device >= kMaxPoolDevices)
        return;
    DevicePool& d = g_pools[device];
    std::lock_guard<std::mutex> guard(d.lock);
    ++d.handles;
    if (d.pool)
        return;
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    unsigned long long keep = kPoolKeep;
    if (cudaMemPoolCreate(&d.pool, &props) != cudaSuccess) {
        d.pool = nullptr;
    } else if (cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess ||
               cudaStreamCreateWithFlags(&d.stream, cudaStreamNonBlocking) != cudaSuccess) {
        cudaMemPoolDestroy(d.pool);
        d.pool = nullptr;
        d.stream = nullptr;
    }
    cudaGetLastError();
}

// The handle's buffers have been freed.
inline void pool_leave(int device)
{
    if (device >= kMaxPoolDevices)
        return;
    DevicePool& d = g_pools[device];
    std::lock_guard<std::mutex> guard(d.lock);
    if (--d.handles == 0 && d.pool) {
        cudaStreamSynchronize(d.stream);         // every release has happened: the memory goes back with the pool
        cudaMemPoolDestroy(d.pool);
        cudaStreamDestroy(d.stream);
        d.pool = nullptr;
        d.stream = nullptr;
    }
}

// `b` is empty; on success it owns `bytes` of device memory that the caller may use on any stream.
inline cudaError_t device_alloc(int device, DevBuf& b, size_t bytes)
{
    cudaMemPool_t pool = nullptr;
    cudaStream_t stream = nullptr;
    if (device < kMaxPoolDevices && bytes <= kPoolLargest) {
        DevicePool& d = g_pools[device];
        std::lock_guard<std::mutex> guard(d.lock);
        pool = d.pool;
        stream = d.stream;
    }
    void* ptr = nullptr;
    cudaError_t e;
    if (!pool) {
        stream = nullptr;
        e = cudaMalloc(&ptr, bytes);
    } else {
        e = cudaMallocFromPoolAsync(&ptr, bytes, pool, stream);
        if (e == cudaSuccess && (e = cudaStreamSynchronize(stream)) != cudaSuccess)
            cudaFreeAsync(ptr, stream);
    }
    if (e != cudaSuccess)
        return e;
    b.ptr = ptr;
    b.bytes = bytes;
    b.stream = stream;
    return cudaSuccess;
}

// (whatever used the memory has finished)
inline cudaError_t device_free(DevBuf& b)
{
    const cudaError_t e = !b.ptr ? cudaSuccess : b.stream ? cudaFreeAsync(b.ptr, b.stream) : cudaFree(b.ptr);
    b = DevBuf();
    return e;
}

} // namespace mem
} // namespace ttc
