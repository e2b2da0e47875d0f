"""The launchers' per-device host state (csrc/hatq_launch.h), compiled with the host compiler
against stand-ins of the CUDA calls: no GPU."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_01653_gb300", "csrc")

PROGRAM = r"""
#include <cassert>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "hatq_launch.h"

// One kernel per pointer: the opt-in the driver would hold, and a call that stalls before it takes effect.
static std::atomic<int> held[2], calls, stall_first, device, fail_next;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void *k, cudaFuncAttribute a, int bytes) {
    assert(a == cudaFuncAttributeMaxDynamicSharedMemorySize);
    const int order = calls.fetch_add(1);
    if (fail_next.exchange(0)) return cudaErrorInvalidValue;
    if (order == 0 && stall_first) std::this_thread::sleep_for(std::chrono::milliseconds(200));
    held[k != nullptr].store(bytes);
    return cudaSuccess;
}

int main() {
    using namespace hatq;
    static SmemOptIn a, b;
    const void *ka = nullptr, *kb = &a;
    // two threads: the first caller's setting lands after the second's, and both may launch any size
    stall_first = 1;
    std::vector<std::thread> t;
    for (int i = 0; i < 2; ++i)
        t.emplace_back([&, i] {
            std::this_thread::sleep_for(std::chrono::milliseconds(50 * i));
            assert(a.set(0, ka) == cudaSuccess);
            assert(i == 0 || held[0] == kMaxDynamicSmem);       // set before this thread launches
        });
    for (auto &x : t) x.join();
    assert(held[0] == kMaxDynamicSmem);
    const int n = calls;
    assert(a.set(0, ka) == cudaSuccess && calls == n);          // kept
    assert(a.set(1, ka) == cudaSuccess && calls == n + 1);      // per device
    fail_next = 1;
    assert(b.set(0, kb) == cudaErrorInvalidValue);              // a failure is reported and not kept
    assert(held[1] == 0 && b.set(0, kb) == cudaSuccess && held[1] == kMaxDynamicSmem);
    int d = -1, sms = 0;
    assert(current_device(&d) == cudaSuccess && d == 0 && device_sms(0, &sms) == cudaSuccess && sms == 152);
    device = kMaxDev;
    assert(current_device(&d) == cudaErrorInvalidDevice);
    std::puts("ok");
}
"""


def test_opt_in_holds_whatever_the_order_of_threads(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = "/usr/local/cuda/include"
    if cxx is None or not os.path.exists(os.path.join(inc, "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, "-I", inc, str(src), "-o", str(exe), "-pthread"], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout == "ok\n"


def test_every_kernel_opts_in_through_it():
    """No launcher sets the attribute to the size of its own launch."""
    for f in glob.glob(os.path.join(CSRC, "*")):
        if os.path.basename(f) != "hatq_launch.h":
            assert not re.search(r"cudaFuncSetAttribute", open(f).read()), f
