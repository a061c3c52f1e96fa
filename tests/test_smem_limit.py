"""The shared limit of a kernel's dynamic shared memory, against a stand-in for the CUDA runtime
that lets a second host thread in between the reading and the setting of the limit (CPU only)."""
import os
import shutil
import subprocess

import pytest

from paper_2511_21660_gb300 import build as lib_build

SOURCE = r"""
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include "smem_limit.h"

static std::atomic<int> limit{49152};   // the kernel's limit, as the stand-in keeps it
static std::atomic<int> sets{0};
static std::atomic<bool> first{true};   // the first reader is slow to act on what it read

extern "C" cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *) {
    a->maxDynamicSharedSizeBytes = limit;
    if (first.exchange(false)) std::this_thread::sleep_for(std::chrono::milliseconds(400));
    return cudaSuccess;
}
extern "C" cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int value) {
    limit = value;
    ++sets;
    return cudaSuccess;
}

int main() {
    const int small = 60000, large = 120000;
    std::thread a([&] { qldpc::allow_smem(nullptr, small); });
    std::this_thread::sleep_for(std::chrono::milliseconds(100));
    std::thread b([&] { qldpc::allow_smem(nullptr, large); });
    a.join();
    b.join();
    if (limit != large) { std::printf("two threads left %d\n", (int)limit); return 1; }
    const int before = sets;
    qldpc::allow_smem(nullptr, small);
    if (limit != large || sets != before) { std::printf("lowered to %d\n", (int)limit); return 1; }
    return 0;
}
"""


def test_limit_is_raised_as_one_step_and_never_lowered(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(lib_build.nvcc()))),
                           "include")
    src, exe = tmp_path / "limit.cpp", tmp_path / "limit"
    src.write_text(SOURCE)
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", lib_build.CSRC, "-I", include,
                    str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
