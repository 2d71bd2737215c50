"""buffers.h against a fake CUDA runtime on the host: after a growth in which any
one allocation failed, the next growth -- of any size, the old one included --
finds the capacity at zero and leaves every buffer allocated and large enough."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1811_02761_gb300", "csrc")

HARNESS = r"""
#include "buffers.h"
#include <cstdio>
#include <cstdlib>
static int calls = 0, fail_at = -1, live = 0;
extern "C" {
cudaError_t cudaMalloc(void **p, size_t b) {
    if (calls++ == fail_at) return cudaErrorMemoryAllocation;
    live++;
    *p = malloc(b);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) { live--; free(p); return cudaSuccess; }
}
using namespace nb;
#define CHECK(c) do { if (!(c)) { printf("fail at %d, line %d: %s\n", k, __LINE__, #c); return 1; } } while (0)
int main() {
    for (int k = 0; k < 3; k++)
        for (long next = 50; next <= 200; next += 50) {
            DevBuf a, b, c;
            long cap = 0;
            int inits = 0;
            auto want = [&](long n) {
                if (n <= cap) return cudaSuccess;
                const cudaError_t e = grow(cap, n, {{&a, (size_t)n * 8}, {&b, (size_t)n * 4}, {&c, (size_t)n}});
                if (e == cudaSuccess) inits++;
                return e;
            };
            fail_at = -1;
            CHECK(want(100) == cudaSuccess && cap == 100 && inits == 1);
            calls = 0;
            fail_at = k;
            CHECK(want(150) == cudaErrorMemoryAllocation && cap == 0 && inits == 1);
            fail_at = -1;
            CHECK(want(next) == cudaSuccess && cap == next && inits == 2);
            CHECK(a.p && b.p && c.p && live == 3);
            CHECK(a.bytes >= (size_t)next * 8 && b.bytes >= (size_t)next * 4 && c.bytes >= (size_t)next);
            for (DevBuf *d : {&a, &b, &c}) cudaFree(d->p);
        }
    return 0;
}
"""


def test_growth_after_a_failed_allocation(tmp_path):
    gxx, cuda = shutil.which("g++"), "/usr/local/cuda/include"
    if not gxx or not os.path.isdir(cuda):
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path / "harness.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "harness")
    r = subprocess.run([gxx, "-std=c++17", f"-I{CSRC}", f"-I{cuda}", str(src), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
