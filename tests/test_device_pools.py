"""The library's memory pools against a fake CUDA runtime, without a GPU: what
an allocation that finds no memory does before it is given up."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

# A device of `room` bytes. A block freed in stream order stays taken until a
# device synchronisation (its stream's work is in flight); then it is unused
# pool memory, which trimming gives back.
FAKE = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include <string>
#include "device_pools.cuh"
using namespace krl;
static size_t room = 100, pending = 0, unused_ = 0;
static bool capturing = false;
static std::string calls;
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) { static char h[2]; static int n = 0; *p = (cudaMemPool_t)(h + n++); return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { calls += "t"; room += unused_; unused_ = 0; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { calls += "w"; unused_ += pending; pending = 0; return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c)
{
    *c = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t)
{
    calls += "a";
    if (n > room) return cudaErrorMemoryAllocation;
    room -= n;
    *p = &room;
    return cudaSuccess;
}
}
int main(int argc, char** argv)
{
    const bool scratch = atoi(argv[1]), cap = atoi(argv[2]);
    const size_t held = atoi(argv[3]), want = atoi(argv[4]);
    void* p = nullptr;
    if (pool_alloc(&p, held, true, nullptr) != cudaSuccess) return 1;
    pending = held;                 // freed behind work in flight
    capturing = cap;
    calls.clear();
    if (argc > 5) {
        const cudaError_t t = pools_trim();
        printf("%d %s%zu\n", (int)t, calls.c_str(), room);
        return 0;
    }
    const cudaError_t e = pool_alloc(&p, want, scratch, nullptr);
    printf("%d %s\n", (int)e, calls.c_str());
    return 0;
}
"""


@pytest.fixture(scope="module")
def alloc(tmp_path_factory):
    if not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime_api.h")):
        pytest.skip("no CUDA headers")
    d = tmp_path_factory.mktemp("pools")
    (d / "p.cpp").write_text(FAKE)
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(CUDA, "include"), "-I",
                           os.path.join(ROOT, "paper_2608_09340_gb300", "csrc"), str(d / "p.cpp"), "-o", str(d / "p")])

    def run(scratch, capturing, held, want, *trim):
        args = [str(int(v)) for v in (scratch, capturing, held, want, *trim)]
        out = subprocess.check_output([str(d / "p"), *args], text=True)
        e, calls = out.split()
        return int(e), calls
    return run


def test_first_try(alloc):
    assert alloc(False, False, 50, 50) == (0, "a")


def test_kept_memory_waits_for_frees_in_flight(alloc):
    assert alloc(False, False, 80, 50) == (0, "awtta")


def test_kept_memory_that_is_not_there(alloc):
    assert alloc(False, False, 80, 101) == (2, "awtta")         # cudaErrorMemoryAllocation


def test_scratch_and_captures_do_not_wait(alloc):
    assert alloc(True, False, 80, 50) == (2, "atta")
    assert alloc(False, True, 80, 50) == (2, "atta")


def test_trim_gives_everything_back(alloc):
    assert alloc(False, False, 80, 0, 1) == (0, "wtt100")
