"""The double-word operations of csrc/dword.cuh on the CPU: the header is plain
IEEE arithmetic, so a host compiler runs it with the intrinsics replaced."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_02207_gb300", "csrc")

STUB = """
#pragma once
#include <cmath>
#define __device__
#define __forceinline__ inline
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
inline float __double2float_rn(double x) { return (float)x; }
"""

# argv: number of products. Prints the rms errors, relative to the terms' magnitudes, of the sum of the products by
# dw_add_mul (n products) and by dw_dot2 (pairs), each with that of dw_add and dw_mul spelt out.
MAIN = """
#include <cstdio>
#include <cstdlib>
#include <random>
#include "dword.cuh"
using namespace gbfmm;
int main(int, char** argv) {
    const int n = std::atoi(argv[1]);
    std::mt19937_64 rng(n);
    auto number = [&] {  // uniform on [-1, 1), times a power of two
        const double x = (double)(int64_t)rng() * 0x1p-63;
        return dw_from(std::ldexp(x, (int)(rng() % 7) - 3));
    };
    long double e[4] = {0, 0, 0, 0};
    for (int t = 0; t < 200000; ++t) {
        dw a = dw_make(0.0f, 0.0f), ar = a, d = a, dr = a, px = a, py = a;
        long double exact = 0, size = 0;
        for (int k = 0; k < n; ++k) {
            const dw x = number(), y = number();
            const long double v = ((long double)x.hi + x.lo) * ((long double)y.hi + y.lo);
            exact += v;
            size += std::fabs(v);
            a = dw_add_mul(a, x, y);
            ar = dw_add(ar, dw_mul(x, y));
            if (k % 2) {
                d = dw_add(d, dw_dot2(px, py, x, y));
                dr = dw_add(dr, dw_add(dw_mul(px, py), dw_mul(x, y)));
            }
            px = x;
            py = y;
        }
        if (n % 2) {
            d = dw_add_mul(d, px, py);
            dr = dw_add(dr, dw_mul(px, py));
        }
        const dw r[4] = {a, ar, d, dr};
        for (int i = 0; i < 4; ++i) {
            const long double q = ((long double)r[i].hi + r[i].lo - exact) / size;
            e[i] += q * q;
        }
    }
    for (int i = 0; i < 4; ++i) std::printf("%.9Le\\n", std::sqrt(e[i] / 200000));
}
"""


@pytest.mark.parametrize("n", [1, 2, 3, 4, 8, 13])
def test_sums_of_products_are_as_exact_as_products_and_sums(tmp_path, n):
    """Sums of up to 13 products are what the swaps and the z-shift of a translation take. The sampling
    error of the two rms values, which see the same numbers, is far below 1 %."""
    (tmp_path / "cuda_runtime.h").write_text(STUB)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "main"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", str(tmp_path), "-I", CSRC,
                    str(tmp_path / "main.cpp"), "-o", str(exe)], check=True)
    e = [float(v) for v in subprocess.run([str(exe), str(n)], check=True, capture_output=True, text=True).stdout.split()]
    assert e[0] <= 1.01 * e[1] and e[2] <= 1.01 * e[3]
    assert max(e) < 4 * 2.0**-48  # a few u^2
