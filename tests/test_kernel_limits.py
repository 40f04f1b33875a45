"""Shared-memory limits of kernels belong to a device: every context raises them for its own, and once.  The host code is compiled with a
runtime call that only writes down what it was asked, so that a second device needs no GPU."""
import os
import shutil
import subprocess

import pytest

from paper_2202_02365_b200 import build

SOURCE = r"""
#include <cuda_runtime.h>
#include <cstdarg>
#include <cstdio>
#include <map>
static std::map<int, std::map<const void*, int>> asked;   // device -> kernel -> calls
static int current = 0;
static cudaError_t write_down(const void* kernel, cudaFuncAttribute, int) { ++asked[current][kernel]; return cudaSuccess; }
#define cudaFuncSetAttribute(kernel, attribute, value) write_down((const void*)(kernel), attribute, value)
#include "mg_sample.cu"

int mg_fail(mg_ctx*, int code, const char*, ...) { return code; }
int mg_cuda_fail(mg_ctx*, cudaError_t, const char*) { return MG_ERR_CUDA; }
void mg_prof_begin(mg_ctx*, int) {}
void mg_prof_end(mg_ctx*, int, int64_t) {}

int main() {
    for (int round = 0; round < 2; ++round)
        for (int device = 0; device < 2; ++device) {
            static mg_ctx contexts[2];
            current = device;
            contexts[device].device = device;
            if (sample_kernel_limits(&contexts[device]) != MG_OK) return 1;
        }
    for (int device = 0; device < 2; ++device) {
        if (asked[device].size() != 3) { printf("device %d: %zu kernels\n", device, asked[device].size()); return 2; }
        for (auto& k : asked[device]) if (k.second != 1) { printf("device %d: raised %d times\n", device, k.second); return 3; }
    }
    return 0;
}
"""


def test_sampler_limits_are_raised_on_every_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    source = tmp_path / "limits.cu"
    source.write_text(SOURCE)
    program = str(tmp_path / "limits")
    made = subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-O0", "-Xptxas", "-O0", "-Xcompiler", "-w",
                           "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"), str(source), "-o", program], capture_output=True, text=True)
    assert made.returncode == 0, made.stderr[-2000:]
    ran = subprocess.run([program], capture_output=True, text=True)
    assert ran.returncode == 0, ran.stdout
