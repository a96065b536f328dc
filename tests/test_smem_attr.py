"""The permission for large dynamic shared memory is asked for once per kernel AND device: the helper against a fake of the CUDA
runtime with three devices and several threads, and no launch that goes past it."""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1611_07151_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <set>
#include <thread>
#include <utility>
#include <vector>
#include "smem_attr.h"

static thread_local int device = 0;
static std::mutex mu;
static std::multiset<std::pair<int, const void*>> asked;
static int fail = 0;

extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v)
{
    if (a != cudaFuncAttributeMaxDynamicSharedMemorySize || v != 100000) return cudaErrorInvalidValue;
    std::lock_guard<std::mutex> lock(mu);
    if (fail) { --fail; return cudaErrorUnknown; }
    asked.insert({device, f});
    return cudaSuccess;
}

int main()
{
    static char k1, k2;
    static sqn::SmemAttr a1, a2;
    fail = 1;
    if (a1.allow(&k1, 100000) != cudaErrorUnknown) return 1;        // a failure is reported and not remembered
    for (int turn = 0; turn < 2; ++turn)
        for (device = 0; device < 3; ++device) {
            if (a1.allow(&k1, 100000) != cudaSuccess || a2.allow(&k2, 100000) != cudaSuccess) return 2;
            if (asked.count({device, &k1}) != 1 || asked.count({device, &k2}) != 1) return 3;
        }
    static sqn::SmemAttr a3;
    static char k3;
    std::vector<std::thread> threads;
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([t] {
            device = t & 1;
            for (int i = 0; i < 1000; ++i) {
                if (a3.allow(&k3, 100000) != cudaSuccess) std::abort();
                std::lock_guard<std::mutex> lock(mu);
                if (!asked.count({device, &k3})) std::abort();      // never skipped on a device before it was set there
            }
        });
    for (auto& t : threads) t.join();
    puts("ok");
    return 0;
}
"""


def test_asked_for_once_per_kernel_and_device(tmp_path):
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc"))
    if nvcc is None:
        pytest.skip("no CUDA toolkit")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    src, exe = tmp_path / "fake.cpp", tmp_path / "fake"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, "-I", include, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout == "ok\n"


def test_no_launch_goes_past_it():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h")):
        if os.path.basename(path) != "smem_attr.h":
            assert not re.search(r"cudaFuncSetAttribute\s*\(", open(path).read()), path
