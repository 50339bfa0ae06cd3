"""Per-device settings (csrc/qmc_device_once.h) on the CPU, with a fake of the
runtime call that sets a kernel's shared memory limit: once for each current
device, again after a failure, also from several threads; and that no kernel
keeps one process-wide answer."""
import os
import re
import shutil
import subprocess

import pytest

from test_kernel_math_host import CSRC

SRC = r"""
#include <cstdio>
#include <thread>
#include <vector>
#define __CUDACC__
enum cudaError_t { cudaSuccess = 0, cudaErrorUnknown = 1 };
enum cudaFuncAttribute { cudaFuncAttributeMaxDynamicSharedMemorySize };
static thread_local int g_dev = 0;
static int g_limit[128], g_calls[128];
static bool g_fail = false;
static cudaError_t cudaGetDevice(int *d) { *d = g_dev; return cudaSuccess; }
template <class K> cudaError_t cudaFuncSetAttribute(K *, cudaFuncAttribute, int bytes) {
    __sync_fetch_and_add(&g_calls[g_dev], 1);
    if (g_fail) return cudaErrorUnknown;
    g_limit[g_dev] = bytes;
    return cudaSuccess;
}
#include "qmc_device_once.h"
static void kernel(int) {}
#define CHECK(c) if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; }
int main() {
    std::atomic<uint64_t> done{0};
    g_fail = true;
    CHECK(!qmc_allow_smem(done, kernel, 7));
    g_fail = false;                                    // a failure is not kept
    for (int dev : {0, 1, 63, 0, 1, 63, 64, 64}) {
        g_dev = dev;
        CHECK(qmc_allow_smem(done, kernel, 1000 + dev));
        CHECK(g_limit[dev] == 1000 + dev);
    }
    CHECK(g_calls[0] == 2 && g_calls[1] == 1 && g_calls[63] == 1 && g_calls[64] == 2);
    std::atomic<uint64_t> other{0};                    // another kernel's state
    std::vector<std::thread> t;
    bool ok[16] = {};
    for (int i = 0; i < 16; ++i)
        t.emplace_back([&, i] { g_dev = i % 4; ok[i] = qmc_allow_smem(other, kernel, 5) && g_limit[i % 4] == 5; });
    for (auto &x : t) x.join();
    for (bool o : ok) CHECK(o);
    CHECK(other.load() == 15);
    return 0;
}
"""


def test_once_per_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    (tmp_path / "t.cpp").write_text(SRC)
    subprocess.run([cxx, "-O1", "-std=c++17", "-pthread", "-I", CSRC, str(tmp_path / "t.cpp"), "-o",
                    str(tmp_path / "t")], check=True, capture_output=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_every_limit_is_set_per_device():
    for f in os.listdir(CSRC):
        if f.endswith((".cu", ".cuh", ".cpp", ".h")) and f != "qmc_device_once.h":
            text = open(os.path.join(CSRC, f)).read()
            assert not re.search(r"cudaFuncSetAttribute\(", text), f
