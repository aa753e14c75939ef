"""The contraction's FP64 division (csrc/ivs_div.cuh) compiled for the host: its integer arithmetic is
defined for every pair of operands (signed overflow traps), and its quotients equal the machine's in
the three roundings."""

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cfenv>
#include <cmath>
#include <cstdio>
#include <cstring>
#define IVS_HD
#define __device__
#define __forceinline__ inline
#include "division_operands.h"
static long long __double_as_longlong(double d) { long long u; std::memcpy(&u, &d, 8); return u; }
static double __longlong_as_double(long long u) { double d; std::memcpy(&d, &u, 8); return d; }
static float __uint2float_rn(unsigned x) { return (float)x; }
static float __int2float_rn(int x) { return (float)x; }
static int __float2int_rn(float x) { return (int)std::rint(x); }
static double rounded(double a, double b, int mode) {
    std::fesetround(mode);
    volatile double x = a, y = b, q = x / y;
    std::fesetround(FE_TONEAREST);
    return q;
}
static double __ddiv_rn(double a, double b) { return rounded(a, b, FE_TONEAREST); }
static double __ddiv_rd(double a, double b) { return rounded(a, b, FE_DOWNWARD); }
static double __ddiv_ru(double a, double b) { return rounded(a, b, FE_UPWARD); }
#include "ivs_div.cuh"

static bool same(double x, double y) { return std::memcmp(&x, &y, 8) == 0 || (x != x && y != y); }

int main() {
    long bad = 0;
    for (int k = 0; k < kClasses; k++)
        for (uint64_t i = 0; i < 400000; i++) {
            uint64_t ua, ub;
            operands(k, i, ua, ub);
            const double a = __longlong_as_double((long long)ua), b = __longlong_as_double((long long)ub);
            bad += !same(ivs::div_exact<ivs::DIV_RN>(a, b), __ddiv_rn(a, b));
            bad += !same(ivs::div_exact<ivs::DIV_RD>(a, b), __ddiv_rd(a, b));
            bad += !same(ivs::div_exact<ivs::DIV_RU>(a, b), __ddiv_ru(a, b));
        }
    std::printf("%ld\n", bad);
    return 0;
}
"""


def test_division_on_the_host(tmp_path):
    source, program = tmp_path / "division.cpp", tmp_path / "division"
    source.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-frounding-math", "-ffp-contract=off", "-fsanitize=undefined",
                    "-fsanitize-undefined-trap-on-error", "-I", os.path.join(ROOT, "tests"),
                    "-I", os.path.join(ROOT, "paper_1802_00330_gb300", "csrc"), "-o", str(program), str(source)], check=True)
    run = subprocess.run([str(program)], capture_output=True, text=True)
    assert run.returncode == 0, "trapped: undefined integer arithmetic"
    assert int(run.stdout) == 0
