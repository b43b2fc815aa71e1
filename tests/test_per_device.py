"""Per-device set-up of kernels (csrc/per_device.h) against a CUDA runtime of two devices that only
counts calls: attributes and SM counts are asked for once on each device, from any thread, again after
a failure; and no other source sets a function attribute."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1811_03339_gb300", "csrc")

RUNTIME = r"""
#pragma once
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1 };
enum { cudaDevAttrMultiProcessorCount = 16 };
enum { cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
extern thread_local int t_dev;
extern int n_set[2], n_count[2], fail_next;
inline cudaError_t cudaGetDevice(int *d) { *d = t_dev; return cudaSuccess; }
inline cudaError_t cudaDeviceGetAttribute(int *v, int, int d) {
    n_count[d]++;
    *v = 100 + d;
    return cudaSuccess;
}
inline cudaError_t cudaFuncSetAttribute(const void *, int, int) {
    if (fail_next) { fail_next = 0; return cudaErrorInvalidValue; }
    n_set[t_dev]++;
    return cudaSuccess;
}
"""
MAIN = r"""
#include "per_device.h"
#include <stdio.h>
#include <thread>
#include <vector>
thread_local int t_dev = 0;
int n_set[2], n_count[2], fail_next;
static void ka() {}
static void kb() {}
int main() {
    fail_next = 1;
    if (fem3::device_smem((const void *)ka, 1 << 17) == cudaSuccess) return 1;
    std::vector<std::thread> ts;
    for (int i = 0; i < 16; i++)
        ts.emplace_back([i] {
            t_dev = i & 1;
            for (int k = 0; k < 1000; k++) {
                int s = 0;
                if (fem3::device_sms(&s) != cudaSuccess || s != 100 + t_dev) _Exit(2);
                if (fem3::device_smem((const void *)ka, 1 << 17) != cudaSuccess) _Exit(3);
                if (fem3::device_smem((const void *)kb, 1 << 16) != cudaSuccess) _Exit(4);
            }
        });
    for (auto &t : ts) t.join();
    printf("%d %d %d %d\n", n_set[0], n_set[1], n_count[0], n_count[1]);
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_once_per_device(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "main.cpp").write_text('#include <stdlib.h>\n' + MAIN)
    exe = tmp_path / "main"
    subprocess.run(["g++", "-std=c++17", "-pthread", f"-I{tmp_path}", f"-I{CSRC}",
                    str(tmp_path / "main.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    assert out.split() == ["2", "2", "1", "1"]


def test_attributes_are_set_in_one_place():
    users = [f for f in os.listdir(CSRC) if re.search(r"\bcudaFuncSetAttribute\b",
                                                      open(os.path.join(CSRC, f)).read())]
    assert users == ["per_device.h"]
