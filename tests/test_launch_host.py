"""Launch set-up per device, on the CPU: kns_launch.h compiled against a recorded stand-in for the CUDA runtime."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <cstdio>
#include "kns_launch.h"
static int dev = 0, asked = 0, limit[64];  // the current device, occupancy queries, each device's limit
extern "C" cudaError_t cudaGetDevice(int *d) { *d = dev; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void *, enum cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limit[dev] = v;
    return cudaSuccess;
}
extern "C" cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int, size_t) {
    ++asked;
    *n = 3 + dev;  // devices may differ
    return cudaSuccess;
}
static void kernel() {}
int main() {
    static kns::PerDevice cache;
    const int order[] = {0, 0, 1, 0, 1, 63, 63};  // 63: past the devices whose answers are kept
    for (int d : order) {
        int n = 0;
        dev = d;
        if (kns::resident_blocks(kernel, 128, 70000, cache, n) != cudaSuccess) return 1;
        std::printf("%d %d %d\n", n, limit[d], asked);
    }
    return 0;
}
"""


def test_every_device_gets_a_kernels_shared_memory_limit(tmp_path):
    """A launch on a device is refused unless that device was given the kernel's limit."""
    cuda = next((p for p in ("/usr/local/cuda/include", os.environ.get("CUDA_HOME", "") + "/include")
                 if os.path.exists(os.path.join(p, "cuda_runtime.h"))), None)
    gxx = shutil.which("g++")
    if cuda is None or gxx is None:
        pytest.skip("no CUDA headers or no g++")
    src, exe = tmp_path / "launch.cpp", tmp_path / "launch"
    src.write_text(SOURCE)
    csrc = os.path.join(ROOT, "paper_2206_10885_gb300", "csrc")
    subprocess.run([gxx, "-std=c++17", "-I", cuda, "-I", csrc, str(src), "-o", str(exe)], check=True)
    got = [tuple(map(int, line.split())) for line in subprocess.run([str(exe)], check=True, capture_output=True,
                                                                    text=True).stdout.splitlines()]
    assert got == [(3, 70000, 1), (3, 70000, 1), (4, 70000, 2), (3, 70000, 2), (4, 70000, 2),
                   (66, 70000, 3), (66, 70000, 4)]
