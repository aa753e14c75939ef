"""The contraction's FP64 division (csrc/ivs_div.cuh) against the CUDA library's (GPU), quotient by quotient in
the three roundings, on seeded operands of every kind that it tells apart."""

import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#define IVS_HD __host__ __device__
#include "division_operands.h"
#include "ivs_div.cuh"

__device__ bool same(double x, double y) {
    return __double_as_longlong(x) == __double_as_longlong(y) || (x != x && y != y);
}

__global__ void compare(uint64_t count, unsigned long long *bad) {
    for (int k = 0; k < kClasses; k++)
        for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (uint64_t)gridDim.x * blockDim.x) {
            uint64_t ua, ub;
            operands(k, i, ua, ub);
            const double a = __longlong_as_double((long long)ua), b = __longlong_as_double((long long)ub);
            if (!same(ivs::div_exact<ivs::DIV_RN>(a, b), __ddiv_rn(a, b))) atomicAdd(bad + 3 * k, 1ull);
            if (!same(ivs::div_exact<ivs::DIV_RD>(a, b), __ddiv_rd(a, b))) atomicAdd(bad + 3 * k + 1, 1ull);
            if (!same(ivs::div_exact<ivs::DIV_RU>(a, b), __ddiv_ru(a, b))) atomicAdd(bad + 3 * k + 2, 1ull);
        }
}

int main() {
    unsigned long long *bad, host[3 * kClasses];
    if (cudaMalloc(&bad, sizeof(host)) != cudaSuccess || cudaMemset(bad, 0, sizeof(host)) != cudaSuccess) return 1;
    compare<<<608, 256>>>(1ull << 25, bad);
    if (cudaMemcpy(host, bad, sizeof(host), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    for (int k = 0; k < 3 * kClasses; k++) std::printf("%llu ", host[k]);
    return 0;
}
"""


def test_quotients_equal_the_library(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    source, program = tmp_path / "division.cu", tmp_path / "division"
    source.write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-O3", "-fmad=false", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "tests"), "-I", os.path.join(ROOT, "paper_1802_00330_gb300", "csrc"),
                    "-o", str(program), str(source)], check=True)
    run = subprocess.run([str(program)], capture_output=True, text=True, timeout=120)
    assert run.returncode == 0
    assert [int(x) for x in run.stdout.split()] == [0] * 21
