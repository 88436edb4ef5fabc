"""The buffers' host code (csrc/buffers.h) over a stand-in for the CUDA runtime."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_06955_gb300", "csrc")
RUNTIME = r"""
#include "buffers.h"
#include <cstdio>
#include <cstdlib>
static char place[1 << 20];
static cudaStream_t freed_on;
static size_t limit = sizeof(place);  // larger allocations fail
extern "C" {
// every allocation comes back at the same place, as it may when one that was just freed is replaced
cudaError_t cudaMalloc(void **p, size_t n) { return n > limit ? cudaErrorMemoryAllocation : (*p = place, cudaSuccess); }
cudaError_t cudaFree(void *) { return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *) { return cudaSuccess; }
cudaError_t cudaMallocAsync(void **p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void *, cudaStream_t s) { return freed_on = s, cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *, const void *, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
}
#define CHECK(x) \
    if (!(x)) { \
        printf("line %d: %s\n", __LINE__, #x); \
        exit(1); \
    }
"""


def run(tmp_path, main):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = "/usr/local/cuda/include"
    if cxx is None or not os.path.exists(os.path.join(inc, "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or no CUDA headers")
    src, exe = tmp_path / "buffers.cpp", tmp_path / "buffers"
    src.write_text(RUNTIME + "int main() {" + main + "}")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-I", inc, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_new_memory_is_told_by_the_allocation_not_by_its_address(tmp_path):
    run(tmp_path, r"""
    DevBuf b;
    bool fresh = false;
    CHECK(b.ensure(1000, &fresh) == cudaSuccess && fresh);
    const void *before = b.p;
    CHECK(b.ensure(900, &fresh) == cudaSuccess && !fresh);
    CHECK(b.ensure(b.cap, &fresh) == cudaSuccess && !fresh);
    CHECK(b.ensure(b.cap + 1, &fresh) == cudaSuccess && fresh && b.p == before);  // grown in place: its end is new
    b.release();
    CHECK(b.ensure(10, &fresh) == cudaSuccess && fresh && b.p == before);
    CHECK(b.ensure(2 << 20, &fresh) != cudaSuccess && b.p == nullptr);
    CHECK(b.ensure(10, &fresh) == cudaSuccess && fresh);
    """)


def test_memory_still_being_written_is_freed_in_its_writers_order(tmp_path):
    run(tmp_path, r"""
    const cudaStream_t writer = (cudaStream_t)0x1234;
    DevBuf b;
    CHECK(b.alloc_pooled(1000, writer) == cudaSuccess);
    b.release();  // an update that failed half-way: kernels on `writer` may be at it
    CHECK(freed_on == writer);
    CHECK(b.alloc_pooled(1000, writer) == cudaSuccess);
    b.settle();  // written and published; the last reader lets go, on whatever thread
    b.release();
    CHECK(freed_on == cudaStreamPerThread);
    CHECK(b.alloc_pooled(2000, writer) == cudaSuccess && b.alloc_pooled(1000, writer) == cudaSuccess);
    CHECK(freed_on == writer);
    """)
