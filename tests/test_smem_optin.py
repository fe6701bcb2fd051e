"""The opt-in to large dynamic shared memory (csrc/smem_optin.cuh): whatever threads
and devices launch a kernel, and however their sizes differ, its limit on a device is
in place before a launch there and never drops below an earlier one.

No GPU: the header is compiled against a stand-in for the four runtime calls it makes."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2209_05934_gb300", "csrc")

RUNTIME = r"""
#pragma once
#include <stddef.h>
#include <atomic>
typedef int cudaError_t;
enum { cudaSuccess = 0, cudaErrorInvalidValue = 1 };
enum { cudaDevAttrMaxSharedMemoryPerBlockOptin = 97 };
enum { cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
struct cudaFuncAttributes { size_t sharedSizeBytes; };
inline thread_local int device = 0;
inline std::atomic<int> limit[2][80], drops{0}, sets{0}, failing{0};
inline cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
inline cudaError_t cudaDeviceGetAttribute(int *v, int, int) { *v = 232448; return cudaSuccess; }
void kernel_a();
void kernel_b();
inline int which(const void *f) { return f == (const void *)kernel_b; }
inline cudaError_t cudaFuncGetAttributes(cudaFuncAttributes *a, const void *f) {
    a->sharedSizeBytes = which(f) ? 1088 : 64;
    return cudaSuccess;
}
inline cudaError_t cudaFuncSetAttribute(const void *f, int, int bytes) {
    ++sets;
    if (failing.load()) return cudaErrorInvalidValue;
    if (limit[which(f)][device].exchange(bytes) > bytes) ++drops;
    return cudaSuccess;
}
"""

HARNESS = r"""
#include <stdio.h>
#include <thread>
#include <vector>
#include "smem_optin.cuh"
void kernel_a() {}
void kernel_b() {}
static omm::SmemOptIn a, b;
int main() {
    // a failed opt-in is reported and tried again
    device = 3;
    failing = 1;
    if (a(kernel_a) != cudaErrorInvalidValue) return 1;
    failing = 0;
    if (a(kernel_a) != cudaSuccess || limit[0][3] != 232448 - 64) return 2;
    // threads on several devices: the limit is there when the call returns
    std::atomic<int> bad{0};
    std::vector<std::thread> ts;
    for (int t = 0; t < 16; ++t)
        ts.emplace_back([&, t] {
            for (int i = 0; i < 4000; ++i) {
                device = (t + i) % 4 + (t % 2 ? 62 : 0);   // 0..3 and 62..65
                if (a(kernel_a) != cudaSuccess || limit[0][device] != 232448 - 64) ++bad;
                if (b(kernel_b) != cudaSuccess || limit[1][device] != 232448 - 1088) ++bad;
            }
        });
    for (auto &t : ts) t.join();
    if (bad) return 3;
    if (drops) return 4;
    // once a device is recorded nothing is set again
    device = 1;
    const int before = sets;
    for (int i = 0; i < 100; ++i) a(kernel_a);
    return sets == before ? 0 : 5;
}
"""


def test_limit_holds_for_every_thread_and_device(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "h.cpp").write_text(HARNESS)
    exe = str(tmp_path / "h")
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "h.cpp"),
                    "-o", exe], check=True)
    assert subprocess.run([exe], timeout=60).returncode == 0


def test_every_opt_in_goes_through_the_header():
    """No launcher keeps a limit of its own (a size behind a static is the race above)."""
    for f in sorted(os.listdir(CSRC)):
        if f == "smem_optin.cuh":
            continue
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        assert "cudaFuncSetAttribute" not in text, f
