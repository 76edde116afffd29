"""The library built once more with a cudaMalloc that refuses one call when told to: what an entry point does
when device memory runs out at any of its allocations, without filling the device."""
import ctypes as C
import os
import subprocess

HOOK = """
#pragma once
#include <cuda_runtime.h>
cudaError_t test_malloc(void** p, size_t bytes);
template <class T> static inline cudaError_t test_malloc_t(T** p, size_t bytes) { return test_malloc((void**)p, bytes); }
#define cudaMalloc test_malloc_t
"""
ALLOC = """
#include <cuda_runtime.h>
static long long calls = 0, refuse = -1, sizes[4096];
cudaError_t test_malloc(void** p, size_t bytes) {
    if (calls < 4096) sizes[calls] = (long long)bytes;
    if (calls++ == refuse) return cudaMalloc(p, (size_t)1 << 60);      // refused by the runtime, its last error set
    return cudaMalloc(p, bytes);
}
#define API extern "C" __attribute__((visibility("default")))
API void test_alloc_reset(long long at) { calls = 0; refuse = at; }
API long long test_alloc_calls() { return calls; }
API long long test_alloc_size(long long i) { return sizes[i]; }
"""



def build(d):
    """Compiles the sources that allocate with the refusing cudaMalloc into directory d; returns the library."""
    from paper_1710_07080_gb300 import _build as b
    (d / "hook.h").write_text(HOOK)
    (d / "alloc.cu").write_text(ALLOC)
    flags = [b._nvcc(), *b.ARCH, *b.FLAGS]
    jobs, objs = [], []
    for src in b.SOURCES:
        kept = os.path.join(b.BUILD, src.replace(".cu", ".o"))
        text = open(os.path.join(b.CSRC, src)).read()
        if "cudaMalloc(" not in text and os.path.exists(kept):
            objs.append(kept)
            continue
        objs.append(str(d / src.replace(".cu", ".o")))
        jobs.append(subprocess.Popen([*flags, "-include", str(d / "hook.h"), "-c", os.path.join(b.CSRC, src), "-o",
                                      objs[-1]]))
    jobs.append(subprocess.Popen([*flags, "-c", str(d / "alloc.cu"), "-o", str(d / "alloc.o")]))
    assert all([j.wait() == 0 for j in jobs])
    so = str(d / "libhooked.so")
    subprocess.check_call([*flags[:3], "-shared", "-cudart", "static", "-o", so, *objs, str(d / "alloc.o"), "-lpthread"])
    return so


def install(isira, so, monkeypatch):
    """The package on the library `so`."""
    monkeypatch.setattr(isira, "LIB_PATH", so)
    monkeypatch.setattr(isira, "lib", isira._load())
    isira.lib.test_alloc_reset.argtypes = [C.c_longlong]
    isira.lib.test_alloc_calls.restype = isira.lib.test_alloc_size.restype = C.c_longlong
    isira.lib.test_alloc_size.argtypes = [C.c_longlong]
