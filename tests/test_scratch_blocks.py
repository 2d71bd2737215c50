"""scratch.cu against a fake CUDA runtime on the host: whatever way a call ends,
its stream has been waited for before its page-locked block can be given to
another call or freed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1811_02761_gb300", "csrc")

HARNESS = r"""
#include "scratch.cu"
#include <cstdio>
#include <cstdlib>
static int waits = 0, waits_at_free = -1, host_fails = 0;
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) { *p = (cudaMemPool_t)8; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void **p, size_t b, cudaMemPool_t, cudaStream_t) { *p = malloc(b); return cudaSuccess; }
cudaError_t cudaFreeAsync(void *p, cudaStream_t) { free(p); return cudaSuccess; }
cudaError_t cudaHostAlloc(void **p, size_t b, unsigned) {
    if (host_fails) return cudaErrorMemoryAllocation;
    *p = malloc(b);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { waits_at_free = waits; free(p); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { waits++; return cudaSuccess; }
}
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
    char *first = nullptr;
    {   // a call that ends early: its block is given back only after a wait
        nb::Scratch s(nullptr);
        CHECK(s.take(64, 4096) == cudaSuccess);
        first = s.host;
    }
    CHECK(waits == 1);
    {   // the block comes back to the next call, which waits once, in finish
        nb::Scratch s(nullptr);
        CHECK(s.take(64, 4096) == cudaSuccess && s.host == first);
        CHECK(s.finish() == cudaSuccess && waits == 2);
    }
    CHECK(waits == 2);
    {   // a block too large to keep is freed, after the wait
        nb::Scratch s(nullptr);
        CHECK(s.take(0, 16u << 20) == cudaSuccess);
    }
    CHECK(waits == 3 && waits_at_free == 3);
    {   // nothing but device memory
        nb::Scratch s(nullptr);
        CHECK(s.take(64, 0) == cudaSuccess);
    }
    CHECK(waits == 4);
    host_fails = 1;
    {
        nb::Scratch s(nullptr);
        CHECK(s.take(64, 1u << 20) != cudaSuccess && s.host == nullptr);
    }
    nb::Scratch::give_back();
    return 0;
}
"""


def test_no_block_is_returned_in_flight(tmp_path):
    gxx, cuda = shutil.which("g++"), "/usr/local/cuda/include"
    if not gxx or not os.path.isdir(cuda):
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path / "harness.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "harness")
    r = subprocess.run([gxx, "-std=c++17", f"-I{CSRC}", f"-I{cuda}", str(src), "-o", exe, "-lpthread"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
