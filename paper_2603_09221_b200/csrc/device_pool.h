// Device memory of the handles' workspaces: one pool per device, shared by its handles, so that a program that makes handles
// for changing shapes does not pay a cudaMalloc (0.35 ms from 2 MB on, and 0.3 ms for its release) for each.  Host code only.
//
// The pool is made by the first buffer that goes into it and keeps at most kPoolKeep bytes that no handle uses.  When the
// last handle of the device goes, the pool and its stream are destroyed.  Every function may be called from any thread; a
// buffer belongs to one handle, and between that handle's pool_enter and pool_leave the pool cannot go away.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <mutex>

namespace ttc {
namespace mem {

constexpr int kMaxPoolDevices = 64;
constexpr unsigned long long kPoolKeep = 256ull << 20;
// Outside these sizes cudaMalloc is the faster one.  Small buffers (the four status words of n = 64) find room in a block
// that the driver has mapped already: 3 us, where the first buffer of a pool takes 0.22 ms, and making and destroying
// pool and stream 0.25 ms.  Gigabytes are mapped slower by the pool (21 against 13 ms).
constexpr size_t kPoolSmallest = 64ull << 10;
constexpr size_t kPoolLargest = 64ull << 20;

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

// (the device is current, here and below)
inline void pool_enter(int device)
{
    if (device >= kMaxPoolDevices)
        return;
    DevicePool& d = g_pools[device];
    std::lock_guard<std::mutex> guard(d.lock);
    ++d.handles;
}

// (d.lock is held)  Where the pool cannot be made, buffers come from cudaMalloc until a later one makes it; each buffer
// remembers where it came from.
inline void make_pool(DevicePool& d, int device)
{
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
    if (device < kMaxPoolDevices && bytes > kPoolSmallest && bytes <= kPoolLargest) {
        DevicePool& d = g_pools[device];
        std::lock_guard<std::mutex> guard(d.lock);
        if (!d.pool)
            make_pool(d, device);
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
