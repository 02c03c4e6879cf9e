"""Device arrays of results: which device they are freed on and how much of them the
pool holds, with the CUDA runtime replaced by one that writes down the calls (no GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2101_05031_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "common.cuh"

static int current = 0, pool_fails = 0;
static size_t next = 0x1000;
static void* fresh(size_t n) { void* p = (void*)next; next += n; return p; }
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = current; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { current = d; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { printf("sync@%d ", current); return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = fresh(n); printf("malloc@%d ", current); return cudaSuccess; }
cudaError_t cudaFree(void*) { printf("free@%d ", current); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
    if (pool_fails) return cudaErrorMemoryAllocation;
    *p = fresh(n); printf("pool@%d ", current); return cudaSuccess; }
cudaError_t cudaFreeAsync(void*, cudaStream_t s) { printf("unpool@%d/%zu ", current, (size_t)s); return cudaSuccess; }
}
namespace csl {
void keep_pool_memory() {}
void fail(csl_status c, const std::string& m) { throw Error(c, m); }
}
int main() {
    using namespace csl;
    const size_t MB = 1 << 20;
    auto line = [] { printf("| now@%d\n", current); };
    // made on device 1, freed with device 0 current
    current = 1; void* a = result_alloc(0, nullptr, "a"); current = 0; result_free(a); line();
    current = 2; a = result_alloc(MB, nullptr, "a"); result_free(a); result_free(nullptr); line();
    // a large array: cudaMalloc, and cudaFree from anywhere
    current = 1; a = result_alloc(257 * MB, nullptr, "a"); current = 0; result_free(a); line();
    // 1 GiB of them at most in the pool; a freed one makes room
    void* v[5];
    for (void*& p : v) p = result_alloc(256 * MB, nullptr, "v");
    line();
    result_free(v[4]); result_free(v[0]);
    v[0] = result_alloc(200 * MB, nullptr, "v"); v[4] = result_alloc(57 * MB, nullptr, "v");
    line();
    for (void* p : v) result_free(p);
    line();
    // the pool has nothing left: cudaMalloc, and the room is given back
    pool_fails = 1;
    for (int i = 0; i < 8; ++i) result_free(result_alloc(256 * MB, nullptr, "v"));
    line();
    pool_fails = 0; a = result_alloc(256 * MB, nullptr, "v"); result_free(a); line();
}
"""

WANT = """pool@1 sync@1 unpool@1/0 | now@0
pool@2 sync@2 unpool@2/0 | now@2
malloc@1 free@0 | now@0
pool@0 pool@0 pool@0 pool@0 malloc@0 | now@0
free@0 sync@0 unpool@0/0 pool@0 malloc@0 | now@0
sync@0 unpool@0/0 sync@0 unpool@0/0 sync@0 unpool@0/0 sync@0 unpool@0/0 free@0 | now@0
malloc@0 free@0 malloc@0 free@0 malloc@0 free@0 malloc@0 free@0 malloc@0 free@0 malloc@0 free@0 malloc@0 free@0 malloc@0 free@0 | now@0
pool@0 sync@0 unpool@0/0 | now@0
"""


def test_arrays_are_freed_on_their_own_device_and_bounded(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.check_call(["g++", "-std=c++17", "-I", inc, "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                           "-x", "c++", str(tmp_path / "main.cpp"), os.path.join(CSRC, "results.cu"),
                           "-o", exe])
    assert subprocess.check_output([exe]).decode() == WANT
