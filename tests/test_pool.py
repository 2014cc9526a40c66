"""The device-memory pools (csrc/pool.cu, host code) against a fake CUDA runtime that records every
call: two devices are there, so what one GPU cannot show can be checked without any."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_1806_02968_gb300", "csrc", "pool.cu")

FAKE = r'''
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include "%(src)s"
static int cur = 0, made = 0;
static std::map<cudaMemPool_t, bool> alive;        // pools that work
static bool bad_stream(cudaStream_t s) { return s == (cudaStream_t)0xbad; }
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = cur; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { cur = d; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize(void) { printf("sync %%d\n", cur); return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { printf("free %%d %%p\n", cur, p); free(p); return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { printf("default\n"); *p = malloc(n); return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* out, const cudaMemPoolProps* p) {
    *out = (cudaMemPool_t)(size_t)(++made);
    alive[*out] = true;
    printf("create %%d on %%d\n", made, p->location.id);
    return cudaSuccess;
}
cudaError_t cudaMemPoolDestroy(cudaMemPool_t p) {
    printf("destroy %%d\n", (int)(size_t)p);
    return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t p, cudaMemPoolAttr, void*) {
    return alive[p] ? cudaSuccess : cudaErrorInvalidValue;
}
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t p, cudaMemPoolAttr, void* v) {
    memset(v, 0, 8);
    return alive[p] ? cudaSuccess : cudaErrorInvalidValue;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { printf("trim\n"); return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t pool, cudaStream_t s) {
    if (bad_stream(s)) return cudaErrorInvalidResourceHandle;
    if (!alive[pool]) return cudaErrorInvalidValue;
    printf("alloc %%d\n", (int)(size_t)pool);
    *p = malloc(n);
    return cudaSuccess;
}
}
int main() {
    void* p = nullptr;
%(body)s
    return 0;
}
'''


def _run(tmp_path, body):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(inc, "cuda_runtime_api.h")):
        pytest.skip("no CUDA headers")
    c, exe = tmp_path / "t.cpp", tmp_path / "t"
    c.write_text(FAKE % dict(src=SRC, body=body))
    subprocess.run(["g++", "-std=c++17", "-I", inc, "-o", str(exe), str(c)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()


def test_free_waits_for_the_owning_device(tmp_path):
    """A handle of device 1 freed while device 0 is current: device 1 is waited for and the memory
    goes back there; device 0 is current again afterwards."""
    out = _run(tmp_path, '''
    lsq::pool_alloc(&p, 16, (cudaStream_t)0);
    void* q = nullptr;
    cudaSetDevice(1);
    lsq::pool_alloc(&q, 16, (cudaStream_t)0);
    cudaSetDevice(0);
    lsq::pool_free(1, {nullptr, q});
    printf("current %d\\n", cur);
    lsq::pool_free(0, {p});
    lsq::pool_free(1, {nullptr});
''')
    assert out[:4] == ["create 1 on 0", "alloc 1", "create 2 on 1", "alloc 2"]
    assert out[4] == "sync 1" and out[5].startswith("free 1 ") and out[6] == "current 0"
    assert out[7] == "sync 0" and out[8].startswith("free 0 ") and len(out) == 9


def test_a_refused_allocation_keeps_a_live_pool(tmp_path):
    """A caller's bad stream gives the error codes of a dead pool: the pool stays the one it was."""
    out = _run(tmp_path, '''
    for (int i = 0; i < 3; ++i) printf("code %d\\n", (int)lsq::pool_alloc(&p, 16, (cudaStream_t)0xbad));
    lsq::pool_alloc(&p, 16, (cudaStream_t)0);
''')
    assert out == ["create 1 on 0"] + ["code 400"] * 3 + ["alloc 1"]


def test_a_dead_pool_is_replaced_once(tmp_path):
    out = _run(tmp_path, '''
    lsq::pool_alloc(&p, 16, (cudaStream_t)0);
    alive[(cudaMemPool_t)1] = false;
    for (int i = 0; i < 2; ++i) printf("code %d\\n", (int)lsq::pool_alloc(&p, 16, (cudaStream_t)0));
''')
    assert out == ["create 1 on 0", "alloc 1", "create 2 on 0", "alloc 2", "code 0", "alloc 2", "code 0"]
