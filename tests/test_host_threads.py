"""The library's host code under several threads, on the CPU: pcbp_host.cpp built with the thread
sanitizer and a stand-in for the CUDA runtime calls that it makes."""
import os
import subprocess
from pathlib import Path

ROOT = Path(__file__).resolve().parent.parent

RUNTIME = """
#pragma once
enum cudaError_t { cudaSuccess = 0 };
enum cudaDeviceAttr { cudaDevAttrMultiProcessorCount, cudaDevAttrMaxSharedMemoryPerBlockOptin,
                      cudaDevAttrMaxSharedMemoryPerMultiprocessor };
cudaError_t cudaGetDevice(int* dev);
cudaError_t cudaDeviceGetAttribute(int* value, cudaDeviceAttr a, int dev);
"""

PROGRAM = """
#include <cuda_runtime.h>
#include <cstdio>
#include <thread>
#include <vector>
#include "pcbp_internal.h"
thread_local int current = 0;
cudaError_t cudaGetDevice(int* dev) { *dev = current; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* value, cudaDeviceAttr a, int dev) { *value = 100 * (dev + 1) + a; return cudaSuccess; }
int main()
{
    std::vector<std::thread> threads;
    int bad[8] = {};
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([&, t] {
            for (int i = 0; i < 200; ++i) {
                current = (i + t) % 70;
                pcbp::DeviceInfo d;
                if (pcbp::device_info(&d) != PC_OK || d.sms != 100 * (current + 1) || d.smem_optin != d.sms + 1 ||
                    d.smem_per_sm != d.sms + 2) bad[t] = 1;
            }
        });
    for (auto& t : threads) t.join();
    for (int b : bad) if (b) return 1;
    return 0;
}
"""


def test_first_calls_on_a_device_from_several_threads(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "main.cpp").write_text(PROGRAM)
    csrc = ROOT / "paper_1911_08868_gb300" / "csrc"
    exe = tmp_path / "threads"
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-g", "-fsanitize=thread", "-pthread", f"-I{tmp_path}",
                    f"-I{ROOT / 'include'}", f"-I{csrc}", str(tmp_path / "main.cpp"), str(csrc / "pcbp_host.cpp"), "-o", str(exe)],
                   check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr[-4000:]
