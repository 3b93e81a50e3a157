"""A kernel launch that fails reports its own error and leaves none behind for
the calls that follow: launch_if against a fake of the CUDA runtime's two calls."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "launch.cuh"
static cudaError_t next = cudaSuccess, last = cudaSuccess;
static int kernel_arg = 0;
extern "C" cudaError_t CUDARTAPI cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void** args) {
    kernel_arg = *static_cast<int*>(args[0]);
    if (next != cudaSuccess) last = next;
    return next;
}
extern "C" cudaError_t CUDARTAPI cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
static void kernel(int) {}
int main() {
    const int arg = 7;
    next = cudaErrorStreamCaptureInvalidated;
    if (moara::launch(kernel, dim3(1), dim3(32), 0, nullptr, 1, arg) != cudaErrorStreamCaptureInvalidated) return 1;
    if (cudaGetLastError() != cudaSuccess) return 2;
    next = cudaSuccess;
    last = cudaErrorInvalidValue;      // somebody else's error: a launch that succeeds leaves it alone
    if (moara::launch_if(false, kernel, dim3(1), dim3(32), 0, nullptr, 4, arg) != cudaSuccess) return 3;
    if (cudaGetLastError() != cudaErrorInvalidValue) return 4;
    return kernel_arg == 7 ? 0 : 5;
}
"""


def test_failed_launch_leaves_no_error_behind(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-I", inc, "-I", os.path.join(ROOT, "paper_2609_15037_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
