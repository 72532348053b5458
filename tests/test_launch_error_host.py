"""A launch that the CUDA runtime refuses is reported by its own call and leaves nothing behind for the next one: the
launch helpers of csrc/runtime.cuh against a fake runtime that refuses every launch.  Compiled with g++; no GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")
DRIVER = r"""
#include <cstdio>
#include "runtime.cuh"
static cudaError_t g_last = cudaSuccess;
static int g_launches = 0;
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) {
    ++g_launches;
    return g_last = cudaErrorInvalidConfiguration;
}
extern "C" cudaError_t cudaGetLastError() {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
static void kernel(int *, int) {}
int main() {
    int word = 0;
    if (kb::launch_overlapped(kernel, 0u, 32u, size_t(0), cudaStream_t(nullptr), &word, 3) == cudaSuccess) return 1;
    if (g_launches != 1) return 2;
    if (cudaGetLastError() != cudaSuccess) { puts("launch_overlapped left its error behind"); return 3; }
    if (kb::cuda_status(cudaLaunchKernelExC(nullptr, nullptr, nullptr)) != KB_ERR_CUDA) return 4;
    if (cudaGetLastError() != cudaSuccess) { puts("cuda_status left the error behind"); return 5; }
    if (kb::cuda_status(cudaSuccess) != KB_OK) return 6;
    return 0;
}
"""


def test_a_refused_launch_leaves_no_error_behind(tmp_path):
    if not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    src, exe = tmp_path / "driver.cpp", tmp_path / "driver"
    src.write_text(DRIVER)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(CUDA, "include"), "-I",
                    os.path.join(ROOT, "paper_1902_05320_gb300", "csrc"), "-x", "c++", str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
