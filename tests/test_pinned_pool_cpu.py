"""The pool of page-locked staging buffers against a stand-in for the CUDA
runtime: a call never waits for the copies of another call, takes an idle buffer
if there is one, and a device has at most four."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2105_07791_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include <map>
#include "mempool.h"
// stand-in runtime: an event is ready unless its stream is busy
static std::map<cudaEvent_t, cudaStream_t> at;
static std::map<cudaStream_t, bool> busy;
static int waits, allocs, frees, device;
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = malloc(16); ++allocs; return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); ++frees; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)malloc(1); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { at[e] = s; return s == (cudaStream_t)99 ? cudaErrorUnknown : cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t e) { return at.count(e) && busy[at[e]] ? cudaErrorNotReady : cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { waits += at.count(e) && busy[at[e]]; return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { waits += busy[s]; return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t*, const cudaMemPoolProps*) { return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolDestroy(cudaMemPool_t) { return cudaSuccess; }
cudaError_t cudaMallocAsync(void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMallocFromPoolAsync(void**, size_t, cudaMemPool_t, cudaStream_t) { return cudaSuccess; }
}
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
    using namespace ndhss;
    cudaStream_t s1 = (cudaStream_t)1, s2 = (cudaStream_t)2;
    PinnedBuf* a = pinned_acquire();
    CHECK(a && allocs == 1);
    busy[s1] = true;                       // another thread's stream, at work
    pinned_release(a, s1);
    PinnedBuf* b = pinned_acquire();       // not a's, and no wait for it
    CHECK(b && b != a && allocs == 2 && waits == 0);
    pinned_release(b, s2);
    CHECK(pinned_acquire() == b && allocs == 2 && waits == 0);
    PinnedBuf* c = pinned_acquire();
    PinnedBuf* d = pinned_acquire();
    CHECK(c && d && allocs == 4);
    CHECK(pinned_acquire() == nullptr && allocs == 4 && waits == 0);    // four in use or busy: do without
    device = 1;                            // another device has its own
    PinnedBuf* o = pinned_acquire();
    CHECK(o && allocs == 5 && o->dev == 1);
    pinned_release(o, s2);
    device = 0;
    CHECK(pinned_acquire() == nullptr);
    busy[s1] = false;
    CHECK(pinned_acquire() == a);          // its copies have run
    pinned_release(a, (cudaStream_t)99);   // no event could be recorded: given back to the system
    CHECK(frees == 1);
    CHECK(pinned_acquire() != nullptr && allocs == 6 && waits == 0);
    printf("ok\n");
    return 0;
}
"""


def test_a_call_never_waits_for_another_calls_copies(tmp_path):
    cxx, nvcc = shutil.which("g++"), shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "pool"
    r = subprocess.run([cxx, "-std=c++17", "-I", inc, "-I", CSRC, str(tmp_path / "main.cpp"), os.path.join(CSRC, "mempool.cpp"),
                        "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout
