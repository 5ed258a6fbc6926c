"""The scratch pool against a fake of the CUDA calls it makes (no GPU): a pool
serves the context it was made in and no other, also where a new context lies
at the old one's address; their number is bounded; giving back waits for the
device first and makes no pool."""
import ctypes
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1704_02272_gb300", "csrc")

FAKE = r"""
#include <cuda_runtime.h>
#include <string.h>
#include "internal.h"
static void *ctx_ptr = (void *)64;
static unsigned long long ctx_id = 1;
static long pools = 0, synced = 0, trimmed_unsynced = 0, trims = 0, from_default = 0, last_pool = 0;
namespace pfac {
void *current_context() { return ctx_ptr; }
uint64_t current_context_id() { return ctx_id; }
}
extern "C" {
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t *p, const cudaMemPoolProps *) {
    *p = (cudaMemPool_t)(++pools);
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void *) { return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
    *s = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void **p, size_t, cudaMemPool_t pool, cudaStream_t) {
    last_pool = (long)pool;
    *p = (void *)256;
    return cudaSuccess;
}
cudaError_t cudaMallocAsync(void **p, size_t, cudaStream_t) {
    from_default++;
    last_pool = 0;
    *p = (void *)256;
    return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { synced++; return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) {
    trims++;
    if (!synced) trimmed_unsynced++;
    synced = 0;
    return cudaSuccess;
}
void fake_context(unsigned long ptr, unsigned long long id) { ctx_ptr = (void *)ptr; ctx_id = id; }
long fake_alloc() {
    void *p = nullptr;
    pfac::scratch_alloc(&p, 1000, nullptr);
    return last_pool;
}
void fake_trim() { pfac::scratch_trim(); }
long fake_pools() { return pools; }
long fake_trims() { return trims; }
long fake_unsynced() { return trimmed_unsynced; }
}
"""


@pytest.fixture()
def fake(tmp_path):
    sys.path.insert(0, os.path.join(ROOT, "paper_1704_02272_gb300"))
    import build as pfac_build  # the build script, not the package
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(pfac_build.nvcc()))), "include")
    src, lib = tmp_path / "fake.cpp", tmp_path / "libfakepool.so"
    src.write_text(FAKE)
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", f"-I{cuda}", f"-I{CSRC}",
                        str(src), os.path.join(CSRC, "pool.cpp"), "-o", str(lib)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    f = ctypes.CDLL(str(lib))  # a fresh path, so a fresh state
    f.fake_context.argtypes = [ctypes.c_ulong, ctypes.c_ulonglong]
    for n in ("fake_alloc", "fake_pools", "fake_trims", "fake_unsynced"):
        getattr(f, n).restype = ctypes.c_long
    return f


def test_one_pool_for_a_context(fake):
    first = fake.fake_alloc()
    assert first == 1 and [fake.fake_alloc() for _ in range(5)] == [1] * 5


def test_a_new_context_at_the_old_address_gets_its_own(fake):
    first = fake.fake_alloc()
    fake.fake_context(64, 2)
    assert fake.fake_alloc() != first


def test_contexts_in_turn_make_few_pools(fake):
    served = {}
    for i in range(200):
        c = 1 + i % 2
        fake.fake_context(64 * c, c)
        served.setdefault(c, set()).add(fake.fake_alloc())
    assert fake.fake_pools() == 2 and all(len(s) == 1 for s in served.values())
    for c in range(3, 300):  # and contexts that come and go: the default pool in the end
        fake.fake_context(64, c)
        fake.fake_alloc()
    assert fake.fake_pools() <= 8
    fake.fake_context(64, 1)
    assert {fake.fake_alloc()} == served[1]


def test_no_context_no_pool(fake):
    fake.fake_context(0, 0)
    assert fake.fake_alloc() == 0 and fake.fake_pools() == 0


def test_giving_back_waits_and_makes_no_pool(fake):
    fake.fake_trim()
    assert fake.fake_pools() == 0 and fake.fake_trims() == 0
    fake.fake_alloc()
    fake.fake_trim()
    assert fake.fake_trims() == 1 and fake.fake_unsynced() == 0
