"""The workspace pool (csrc/pool.cpp) compiled for the host against a runtime that
only counts: one pool for each context, found again whichever was current in
between, and a new one for a context that was not seen before (a device that was
reset has a new one)."""
from __future__ import annotations

import ctypes as C
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2608_28952_gb300", "csrc")

RUNTIME = r"""
#include <cuda.h>
#include <cuda_runtime.h>
#include "internal.h"
static unsigned long long g_ctx = 1;
static int g_dev = 0, g_made = 0, g_fail = 0;
static CUresult ctx_id(CUcontext, unsigned long long* id) { *id = g_ctx; return CUDA_SUCCESS; }
extern "C" {
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q)
{
    *f = (void*)&ctx_id;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { g_dev = d; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*)
{
    if (g_fail) return cudaErrorMemoryAllocation;
    *p = (cudaMemPool_t)(size_t)(100 + ++g_made);
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t, cudaMemPool_t pool, cudaStream_t) { *p = pool; return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t, cudaStream_t) { *p = (void*)1; return cudaSuccess; }
size_t pool_of(int dev, unsigned long long ctx, int fail)   // the pool that an allocation comes from there (1: the device's own)
{
    g_dev = dev;
    g_ctx = ctx;
    g_fail = fail;
    void* p = nullptr;
    return jac::workspace_alloc(&p, 64, nullptr) == cudaSuccess ? (size_t)p : 0;
}
int pools_made() { return g_made; }
}
"""


@pytest.fixture()
def pool(tmp_path):
    gxx, nvcc = shutil.which("g++"), shutil.which("nvcc")
    if not gxx or not nvcc:
        pytest.skip("no g++ or no CUDA headers")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    (tmp_path / "runtime.cpp").write_text(RUNTIME)
    lib = tmp_path / "pool.so"
    subprocess.run([gxx, "-std=c++17", "-w", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", inc, "-I", CSRC, "-o", str(lib),
                    str(tmp_path / "runtime.cpp"), os.path.join(CSRC, "pool.cpp")], check=True)
    so = C.CDLL(str(lib))
    so.pool_of.restype = C.c_size_t
    so.pool_of.argtypes = [C.c_int, C.c_ulonglong, C.c_int]
    return so


def test_one_pool_for_each_context(pool):
    a, b = pool.pool_of(0, 11, 0), pool.pool_of(0, 12, 0)       # two contexts of one device
    other = pool.pool_of(1, 21, 0)                               # and one of another
    assert len({a, b, other}) == 3 and 1 not in (a, b, other)
    for _ in range(4):
        assert (pool.pool_of(0, 11, 0), pool.pool_of(0, 12, 0), pool.pool_of(1, 21, 0)) == (a, b, other)
    assert pool.pools_made() == 3
    fresh = pool.pool_of(0, 13, 0)                               # after a reset
    assert fresh not in (a, b, other) and pool.pools_made() == 4
    assert pool.pool_of(0, 14, 1) == 1                           # no pool to be had: the device's own
    for i in range(500):                                         # many resets: every allocation is served
        assert pool.pool_of(0, 1000 + i, 0) > 1
    assert pool.pool_of(0, 1499, 0) == pool.pool_of(0, 1499, 0)
