"""Host allocation failures at the C ABI are statuses, never exceptions, and the
bookkeeping of released plans' memory (dkv_pool.cu), against a fake of the CUDA
runtime calls it makes: no GPU."""
import os
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_32663_gb300", "csrc")


def test_pattern_copy_without_host_memory_is_reported():
    """A pattern of 256 MB while the process may grow by 64 MB more."""
    code = textwrap.dedent("""
        import resource
        import numpy as np
        from paper_2609_32663_gb300 import build
        build.build_library()
        import paper_2609_32663_gb300.dkv as dkv
        dkv.lib()
        M = np.zeros((1, 8, 1 << 25), np.uint8)
        sh = dkv.Shape(L=1, H=8, H_kv=1, D=1 << 25, bin_width=1)
        used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
        resource.setrlimit(resource.RLIMIT_AS, (used + (64 << 20), resource.RLIM_INFINITY))
        try:
            dkv.dkv_map_pattern(M, [10], sh, stream=0)
        except dkv.DkvError as e:
            print(e.status == dkv.DKV_ERR_OOM, b"host" in dkv.lib().dkv_last_error())
    """)
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split() == ["True", "True"], (r.returncode, r.stdout, r.stderr[-2000:])


HARNESS = r"""
#include "dkv_pool.cuh"
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <cuda.h>
#include <map>
#include <new>

static bool no_host_memory = false;
void* operator new(std::size_t n)
{
    void* p = no_host_memory ? nullptr : std::malloc(n);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

static char arena[1 << 16];
static int next_ptr = 0, mallocs = 0, frees = 0;
static size_t device_limit = ~size_t(0);
static size_t used = 0;
static std::map<void*, size_t> sizes;
static unsigned long long context_id = 1;

static CUresult fake_current(CUcontext* c) { *c = reinterpret_cast<CUcontext>(1); return CUDA_SUCCESS; }
static CUresult fake_id(CUcontext, unsigned long long* id) { *id = context_id; return CUDA_SUCCESS; }

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n)
{
    if (used + n > device_limit) return cudaErrorMemoryAllocation;
    *p = arena + next_ptr++;
    used += n;
    sizes[*p] = n;
    ++mallocs;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p)
{
    if (!sizes.count(p)) { std::printf("free of an unknown block\n"); std::exit(2); }
    used -= sizes[p];
    sizes.erase(p);
    ++frees;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** fn, unsigned int, unsigned long long,
                                             enum cudaDriverEntryPointQueryResult* q)
{
    *fn = !std::strcmp(name, "cuCtxGetId") ? reinterpret_cast<void*>(fake_id) : reinterpret_cast<void*>(fake_current);
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
}

#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }
constexpr size_t MB = 1 << 20;
using dkv::PlanMemory;
using dkv::plan_alloc;
using dkv::plan_free;

int main()
{
    PlanMemory a, b, c;
    CHECK(plan_alloc(&a, 8 * MB) == cudaSuccess && plan_alloc(&b, 8 * MB) == cudaSuccess);
    // kept while another plan lives, for the same or a somewhat smaller size
    void* pa = a.ptr;
    plan_free(a, true);
    CHECK(frees == 0);
    CHECK(plan_alloc(&c, 3 * MB) == cudaSuccess && c.ptr != pa);  // less than half: not that one
    CHECK(plan_alloc(&a, 5 * MB) == cudaSuccess && a.ptr == pa && a.bytes == 8 * MB);
    // not kept: unfinished work, more than the bound
    plan_free(c, false);
    CHECK(frees == 1);
    CHECK(plan_alloc(&c, 65 * MB) == cudaSuccess);
    plan_free(c, true);
    CHECK(frees == 2);
    // given back for an allocation that does not fit otherwise
    plan_free(a, true);
    device_limit = used + 4 * MB;
    CHECK(plan_alloc(&a, 12 * MB) == cudaSuccess && frees == 3);
    device_limit = ~size_t(0);
    // released from another context: freed, not kept for that context
    context_id = 2;
    plan_free(a, true);
    CHECK(frees == 4);
    CHECK(plan_alloc(&c, 12 * MB) == cudaSuccess);
    plan_free(c, true);  // that context's last plan
    CHECK(frees == 5);
    context_id = 1;
    // no host memory for the bookkeeping: freed, or refused, without an exception
    PlanMemory many[64];
    for (PlanMemory& m : many) CHECK(plan_alloc(&m, 1000) == cudaSuccess);
    no_host_memory = true;
    for (PlanMemory& m : many) plan_free(m, true);
    context_id = 3;
    const cudaError_t e = plan_alloc(&c, 1000);
    no_host_memory = false;
    context_id = 1;
    CHECK(e == cudaErrorMemoryAllocation || e == cudaSuccess);
    // everything is given back with the last plan
    if (e == cudaSuccess) { context_id = 3; plan_free(c, true); context_id = 1; }
    plan_free(b, true);
    CHECK(used == 0 && sizes.empty());
    std::printf("ok\n");
    return 0;
}
"""


def test_released_plan_memory_bookkeeping(tmp_path):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    src, exe = tmp_path / "harness.cpp", tmp_path / "harness"
    src.write_text(HARNESS)
    r = subprocess.run(["g++", "-std=c++17", "-O1", f"-I{CSRC}", f"-I{cuda}/include", "-o", str(exe), str(src), "-x", "c++",
                        os.path.join(CSRC, "dkv_pool.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "ok\n", (r.returncode, r.stdout, r.stderr[-2000:])
