"""Function attributes are set once per device, not once per process (device_once.h): a host program with its
own cudaGetDevice walks several devices and threads, one of them with a call that fails the first time."""
import os
import shutil
import subprocess

from paper_1710_07080_gb300 import _build as b

PROGRAM = """
#include "device_once.h"
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
static thread_local int current = 0;
static thread_local bool broken = false;
extern "C" cudaError_t CUDARTAPI cudaGetDevice(int* d) {
    *d = current;
    return broken ? cudaErrorUnknown : cudaSuccess;
}
int main() {
    isira::PerDeviceOnce once;
    std::vector<int> ran;
    auto on = [&](int dev, cudaError_t e) { current = dev; once([&] { ran.push_back(dev); return e; }); };
    for (int dev : {0, 0, 1, 0, 1, 63}) on(dev, cudaSuccess);
    on(2, cudaErrorUnknown); on(2, cudaSuccess); on(2, cudaSuccess);          // an error is tried again
    on(64, cudaSuccess); on(64, cudaSuccess);                                 // not remembered
    broken = true; on(3, cudaSuccess); broken = false;
    for (int d : ran) std::printf("%d ", d);
    isira::PerDeviceOnce many;
    std::atomic<int> count{0};
    std::vector<std::thread> t;
    for (int i = 0; i < 16; ++i) t.emplace_back([&, i] { current = i % 4; many([&] { ++count; return cudaSuccess; }); });
    for (auto& x : t) x.join();
    std::printf("| %d", count.load());
}
"""


def test_runs_once_on_every_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b._nvcc()))), "include")
    inc = next(d for d in (cuda, "/usr/local/cuda/include") if os.path.exists(os.path.join(d, "cuda_runtime_api.h")))
    subprocess.check_call([shutil.which("g++"), "-std=c++17", "-I", b.CSRC, "-I", inc, str(src), "-o", str(exe), "-lpthread"])
    out = subprocess.check_output([str(exe)], text=True)
    assert out == "0 1 63 2 2 64 64 | 4"


def test_no_function_attribute_is_set_once_per_process():
    for f in os.listdir(b.CSRC):
        assert "call_once" not in open(os.path.join(b.CSRC, f)).read(), f
