"""Set-up of a kernel that belongs to a device (csrc/npw_per_device.h), with a fake cudaGetDevice: once on each
device, once however many threads come first, again after a failure, each time on a device beyond the table."""
import os
import shutil
import subprocess

import pytest

from paper_1602_00182_gb300 import build as B

MAIN = r"""
#include "npw_per_device.h"
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
static thread_local int t_dev = 0;
extern "C" cudaError_t cudaGetDevice(int* d) {
    if (t_dev == 99) return cudaErrorInvalidDevice;
    *d = t_dev;
    return cudaSuccess;
}
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
    static npw::PerDevice<bool> p;
    std::atomic<int> calls[80] = {};
    auto set = [&] { calls[t_dev]++; return cudaSuccess; };
    for (int k = 0; k < 3; ++k)
        for (int d : {0, 1, 63, 0}) { t_dev = d; CHECK(p.once(set) == cudaSuccess); }
    CHECK(calls[0] == 1 && calls[1] == 1 && calls[63] == 1);
    t_dev = 2;
    CHECK(p.once([] { return cudaErrorInvalidValue; }) == cudaErrorInvalidValue);
    CHECK(p.once(set) == cudaSuccess && p.once(set) == cudaSuccess && calls[2] == 1);
    t_dev = 70;
    CHECK(p.once(set) == cudaSuccess && p.once(set) == cudaSuccess && calls[70] == 2);
    t_dev = 99;
    CHECK(p.once([] { return cudaSuccess; }) == cudaErrorInvalidDevice);
    std::vector<std::thread> ts;
    for (int i = 0; i < 16; ++i)
        ts.emplace_back([&, i] { t_dev = 4 + i % 2; for (int k = 0; k < 1000; ++k) p.once(set); });
    for (auto& t : ts) t.join();
    CHECK(calls[4] == 1 && calls[5] == 1);
    struct Size { int allowed = 0; };
    static npw::PerDevice<Size> s;
    int grown = 0;
    for (int d : {0, 1}) {
        t_dev = d;
        for (int want : {10, 5, 20, 20})
            s.with([&](Size& v) { if (want > v.allowed) { v.allowed = want; ++grown; } return cudaSuccess; });
    }
    CHECK(grown == 4);
    std::printf("ok\n");
    return 0;
}
"""


def test_set_up_once_per_device(tmp_path):
    include = os.path.join(os.path.dirname(os.path.dirname(B._nvcc())), "include")
    if not shutil.which("g++") or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    src = tmp_path / "per_device.cc"
    src.write_text(MAIN)
    exe = str(tmp_path / "per_device")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", f"-I{B.CSRC}", f"-I{include}", str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout
