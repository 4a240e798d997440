"""Setups that belong to a device (kernel attributes, cluster sizes): made once on
each, in whatever order the devices and threads come, a failure as well as a
success, and no error left behind.  On the CPU, with the runtime's two calls
played by the test."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#include "ising_per_device.h"
#include <cstdio>
#include <thread>
#include <vector>
static thread_local int current = 0;
static thread_local cudaError_t pending = cudaSuccess;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = current; return current == 99 ? pending = cudaErrorNoDevice : cudaSuccess; }
extern "C" cudaError_t cudaGetLastError() { const cudaError_t e = pending; pending = cudaSuccess; return e; }
#define CHECK(x) if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; }
int main()
{
    static ising::PerDevice<int> p;
    int made[64] = {};
    auto get = [&](int dev) {
        current = dev;
        return p.get([&] { ++made[dev]; if (dev == 2) { pending = cudaErrorInvalidValue; return 0; } return 10 + dev; });
    };
    CHECK(get(0) == 10 && get(1) == 11 && get(0) == 10 && get(1) == 11);
    CHECK(get(2) == 0 && pending == cudaSuccess && get(2) == 0);
    CHECK(made[0] == 1 && made[1] == 1 && made[2] == 1);
    current = 99;
    CHECK(p.get([] { return 5; }) == 0 && pending == cudaSuccess);
    std::vector<std::thread> threads;
    bool ok[16] = {};
    for (int k = 0; k < 16; ++k) threads.emplace_back([&, k] { ok[k] = get(3 + k % 2) == 13 + k % 2; });
    for (auto& t : threads) t.join();
    for (bool b : ok) CHECK(b);
    CHECK(made[3] == 1 && made[4] == 1);
    return 0;
}
"""


def test_made_once_on_each_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    src, exe = tmp_path / "per_device.cpp", tmp_path / "per_device"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", include, "-I",
                    os.path.join(ROOT, "paper_1811_04384_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_no_kernel_setup_is_kept_for_the_process():
    """A function's attributes are set under PerDevice, a handle, or on each call."""
    csrc = os.path.join(ROOT, "paper_1811_04384_gb300", "csrc")
    for fn in sorted(os.listdir(csrc)):
        text = open(os.path.join(csrc, fn)).read()
        assert "static const bool ok =" not in text and "static bool attr_set" not in text, fn
        assert "static const int c = probe" not in text, fn
