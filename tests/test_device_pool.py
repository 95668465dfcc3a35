"""The workspace pool (``csrc/device_pool.h``) against a counting stand-in for the CUDA runtime, on the CPU: memory goes back
to where it came from, nothing is left when the last handle goes, and handles of several threads do not race."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_09221_b200", "csrc")

FAKE_RUNTIME = r"""
#pragma once
#include <cstddef>
#include <cstdlib>
#include <map>
#include <mutex>
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorMemoryAllocation = 2 };
struct FakePool { int unused; };
struct FakeStream { int unused; };
typedef FakePool* cudaMemPool_t;
typedef FakeStream* cudaStream_t;
enum { cudaMemAllocationTypePinned = 1, cudaMemLocationTypeDevice = 1, cudaStreamNonBlocking = 1, cudaMemPoolAttrReleaseThreshold = 4 };
struct cudaMemPoolProps { int allocType; struct { int type, id; } location; };
namespace fake {
inline std::mutex lock;
inline std::map<void*, bool> live;               // allocation -> came from a pool
inline int fail_pools = 0, pools = 0, streams = 0, wrong = 0;
inline cudaError_t take(void** p, size_t n, bool pooled)
{
    std::lock_guard<std::mutex> g(lock);
    *p = std::malloc(n < 64 ? n : 64);
    live[*p] = pooled;
    return cudaSuccess;
}
inline cudaError_t give(void* p, bool pooled)
{
    std::lock_guard<std::mutex> g(lock);
    auto it = live.find(p);
    if (it == live.end() || it->second != pooled) {
        ++wrong;
        return cudaErrorInvalidValue;
    }
    live.erase(it);
    std::free(p);
    return cudaSuccess;
}
} // namespace fake
inline cudaError_t cudaMalloc(void** p, size_t n) { return fake::take(p, n, false); }
inline cudaError_t cudaFree(void* p) { return fake::give(p, false); }
inline cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*)
{
    std::lock_guard<std::mutex> g(fake::lock);
    if (fake::fail_pools > 0) {
        --fake::fail_pools;
        return cudaErrorMemoryAllocation;
    }
    ++fake::pools;
    *p = new FakePool();
    return cudaSuccess;
}
inline cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, int, void*) { return cudaSuccess; }
inline cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
inline cudaError_t cudaMemPoolDestroy(cudaMemPool_t p)
{
    std::lock_guard<std::mutex> g(fake::lock);
    --fake::pools;
    delete p;
    return cudaSuccess;
}
inline cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return fake::take(p, n, true); }
inline cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return fake::give(p, true); }
inline cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, int)
{
    std::lock_guard<std::mutex> g(fake::lock);
    ++fake::streams;
    *s = new FakeStream();
    return cudaSuccess;
}
inline cudaError_t cudaStreamDestroy(cudaStream_t s)
{
    std::lock_guard<std::mutex> g(fake::lock);
    --fake::streams;
    delete s;
    return cudaSuccess;
}
inline cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
"""

DRIVER = r"""
#include "device_pool.h"
#include <cstdio>
#include <cstring>
#include <thread>
#include <vector>
using namespace ttc::mem;

static void handle_life(int rounds)
{
    for (int r = 0; r < rounds; ++r) {
        pool_enter(0);
        DevBuf status, middle, large;
        device_alloc(0, status, kPoolSmallest);
        device_alloc(0, middle, kPoolSmallest + 1);
        device_alloc(0, large, kPoolLargest + 1);
        device_free(status);
        device_free(middle);
        device_free(large);
        pool_leave(0);
    }
}

int main(int, char** argv)
{
    if (!std::strcmp(argv[1], "late_pool")) {            // the first buffer gets no pool, the second one does
        fake::fail_pools = 1;
        pool_enter(0);
        DevBuf a, b;
        device_alloc(0, a, 1 << 20);
        pool_enter(0);
        device_alloc(0, b, 1 << 20);
        device_free(a);
        device_free(b);
        pool_leave(0);
        pool_leave(0);
    } else if (!std::strcmp(argv[1], "threads")) {
        for (int round = 0; round < 200; ++round) {      // two handles, the first attempt at a pool fails
            fake::fail_pools = 1;
            pool_enter(0);
            std::thread worker([] {
                for (int i = 0; i < 20; ++i) {
                    DevBuf b;
                    device_alloc(0, b, 1 << 20);
                    device_free(b);
                }
            });
            std::thread other(handle_life, 3);
            worker.join();
            other.join();
            pool_leave(0);
        }
    } else if (!std::strcmp(argv[1], "no_pool")) {       // handles that need no pool do not make one
        pool_enter(0);
        DevBuf a, b;
        device_alloc(0, a, 16);
        device_alloc(0, b, kPoolLargest + 1);
        std::printf("made=%d ", fake::pools);
        device_free(a);
        device_free(b);
        pool_leave(0);
    } else {                                             // the pool is made again after its last handle went
        handle_life(2);
    }
    std::printf("wrong=%d live=%d pools=%d streams=%d\n", fake::wrong, (int)fake::live.size(), fake::pools, fake::streams);
    return 0;
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("pool")
    (d / "cuda_runtime.h").write_text(FAKE_RUNTIME)
    (d / "driver.cpp").write_text(DRIVER)
    out = {}
    for name, flags in (("plain", []), ("tsan", ["-fsanitize=thread", "-g"])):
        cmd = ["g++", "-std=c++17", "-O1", "-pthread", *flags, "-I", str(d), "-I", CSRC, str(d / "driver.cpp"), "-o", str(d / name)]
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0 or name == "tsan", r.stderr
        out[name] = str(d / name) if r.returncode == 0 else None
    return out


@pytest.mark.parametrize("scenario", ["late_pool", "threads", "again"])
def test_memory_goes_back_where_it_came_from_and_nothing_stays(driver, scenario):
    r = subprocess.run([driver["plain"], scenario], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    assert r.stdout.strip() == "wrong=0 live=0 pools=0 streams=0"


def test_a_pool_is_made_only_for_buffers_that_go_into_it(driver):
    r = subprocess.run([driver["plain"], "no_pool"], capture_output=True, text=True, timeout=120)
    assert r.stdout.strip() == "made=0 wrong=0 live=0 pools=0 streams=0"


def test_handles_of_several_threads_do_not_race(driver):
    if not driver["tsan"]:
        pytest.skip("g++ has no thread sanitizer")
    r = subprocess.run([driver["tsan"], "threads"], capture_output=True, text=True, timeout=300)
    if "ThreadSanitizer: unexpected memory mapping" in r.stderr:
        pytest.skip("the thread sanitizer does not run on this kernel")
    assert r.returncode == 0 and "WARNING" not in r.stderr, r.stderr[-2000:]
    assert "wrong=0" in r.stdout
