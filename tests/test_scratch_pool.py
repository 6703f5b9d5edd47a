"""Bookkeeping of the scratch pool (csrc/scratch.cu) against a stand-in for the
CUDA runtime, compiled with it (no GPU): which pool serves, and that the memory
a pool keeps is given back with the last scene of its context, also where an
earlier context ended with scenes alive, or where two are used in turn."""
import ctypes
import os
import subprocess

import pytest

from paper_1912_12786_gb300 import _build

FAKE = r"""
#include <cuda_runtime_api.h>
namespace vsr {
cudaError_t scratch_alloc(void** ptr, size_t bytes, cudaStream_t stream);
unsigned long long scratch_scene_created();
void scratch_scene_destroyed(unsigned long long context);
bool current_context_id(unsigned long long* id);
}
static unsigned long long g_ctx = 1;
static int g_device = 0, g_fail = 0, g_pools = 0;
static long g_used = 0;      // pool of the last allocation, 0 the default one
static int g_trims[64];      // per pool: times it was trimmed to zero
extern "C" {
// nvcc registers the unit, which has no kernels
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
    if (g_fail) return cudaErrorNotSupported;
    *p = (cudaMemPool_t)(long)++g_pools;
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t) { ++g_trims[(long)p]; return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void**, size_t, cudaMemPool_t p, cudaStream_t) {
    g_used = (long)p;
    return cudaSuccess;
}
cudaError_t cudaMallocAsync(void**, size_t, cudaStream_t) { g_used = 0; return cudaSuccess; }
void set_context(unsigned long long c) { g_ctx = c; }
void set_device(int d) { g_device = d; }
void set_fail(int f) { g_fail = f; }
long alloc() { void* p; vsr::scratch_alloc(&p, 8, nullptr); return g_used; }
int trims(int p) { return g_trims[p]; }
unsigned long long created() { return vsr::scratch_scene_created(); }
void destroyed(unsigned long long c) { vsr::scratch_scene_destroyed(c); }
}
bool vsr::current_context_id(unsigned long long* id) { *id = g_ctx; return g_ctx != 0; }
"""


@pytest.fixture()
def pool(tmp_path):
    (tmp_path / "fake.cpp").write_text(FAKE)
    lib = str(tmp_path / "libfake.so")
    subprocess.run([_build._nvcc(), *_build.nvcc_flags(), "-shared", "-cudart", "none",
                    "-Xlinker", "-Bsymbolic", str(tmp_path / "fake.cpp"),
                    os.path.join(_build.CSRC, "scratch.cu"), "-o", lib], check=True)
    c = ctypes.CDLL(lib)
    for f in (c.created, c.alloc):
        f.restype = ctypes.c_uint64
    c.set_context.argtypes = c.destroyed.argtypes = [ctypes.c_uint64]
    return c


def test_pool_follows_contexts_and_scenes(pool):
    c = pool
    assert c.alloc() == 0  # no scene yet: the default pool
    a, b = c.created(), c.created()
    assert c.alloc() == 1
    c.destroyed(a)
    assert c.trims(1) == 0
    # the context ends with scene b alive; in the next one scenes come and go
    c.set_context(2)
    assert c.alloc() == 0
    d = c.created()
    assert c.alloc() == 2
    c.destroyed(d)
    assert c.trims(2) == 1
    # ... a late end of b is not the end of a scene of this context
    d, e = c.created(), c.created()
    c.destroyed(b)
    c.destroyed(d)
    assert c.trims(2) == 1
    c.destroyed(e)
    assert c.trims(2) == 2
    # two contexts used in turn keep a pool each
    f = c.created()
    c.set_context(3)
    g = c.created()
    assert c.alloc() == 3
    c.set_context(2)
    assert c.alloc() == 2
    c.destroyed(f)
    assert c.trims(2) == 3 and c.trims(3) == 0
    c.set_context(3)
    assert c.alloc() == 3
    c.destroyed(g)
    assert c.trims(3) == 1
    # no pool to be had: the default one, and counts stay right for a later try
    c.set_context(4)
    c.set_fail(1)
    h = c.created()
    assert c.alloc() == 0
    c.set_fail(0)
    i = c.created()
    assert c.alloc() == 4
    c.destroyed(h)
    assert c.trims(4) == 0
    c.destroyed(i)
    assert c.trims(4) == 1
    # no current context
    c.set_context(0)
    assert c.created() == 0 and c.alloc() == 0
    c.destroyed(0)
