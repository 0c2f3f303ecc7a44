"""The float64 pair kernels' 1/r and 1/r^3 (csrc/rsqrt64.cuh), on the host, from float32 estimates with
errors up to three units in the last place (the hardware's stay within 2.1), against long double: each
result is rounded to 53 bits once before its final multiply-add at the most, so the relative error stays
below half a unit in the last place for 1/r and one for 1/r^3 (2^-53 and 2^-52 of 1..2), plus the series'
rests.  Arguments over the exponents of squared distances, both ends of a binade, estimates with
an all-zero and an all-ones mantissa.

Host only: compiled by the C++ compiler against the CUDA headers; skipped where either is missing."""
import os
import shutil
import subprocess

import pytest

from test_curve_key import CSRC, ROOT, _cuda_include

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cmath>
#include <random>
#include <cuda_runtime.h>
#include "rsqrt64.cuh"
using namespace psum;
int main(int argc, char** argv) {
    const int lo = std::atoi(argv[1]), hi = std::atoi(argv[2]);
    std::mt19937_64 rng(7);
    long double worst1 = 0, worst3 = 0;
    auto check = [&](double r2) {
        const float y0 = (float)(1.0L / sqrtl((long double)estimate_arg(r2)));
        for (int k = -3; k <= 3; ++k) {
            uint32_t yb;
            memcpy(&yb, &y0, 4);
            yb += k;
            const long double t1 = 1.0L / sqrtl((long double)r2), t3 = t1 / (long double)r2;
            worst1 = std::max(worst1, fabsl(rsqrt_refined(r2, yb) / t1 - 1));
            worst3 = std::max(worst3, fabsl(rsqrt3_refined(r2, yb) / t3 - 1));
        }
    };
    for (int i = 0; i < 300000; ++i) check(std::ldexp(1.0 + std::ldexp((double)(rng() >> 12), -52), lo + (int)(rng() % (hi - lo))));
    for (int e = lo; e < hi; ++e)
        for (int k = 0; k < 200; ++k) {
            check(f64_from(f64_bits(std::ldexp(1.0, e)) + k));
            check(f64_from(f64_bits(std::ldexp(2.0, e)) - 1 - k));
            check(f64_from(f64_bits(std::ldexp(1.0, e)) + ((long long)k << 29) - 1));
        }
    printf("%Lg %Lg\n", worst1, worst3);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = _cuda_include()
    if not cxx or not inc:
        pytest.skip("no host C++ compiler or CUDA headers")
    d = tmp_path_factory.mktemp("rsqrt")
    src, exe = d / "rsqrt.cpp", d / "rsqrt"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", inc, "-I", os.path.join(ROOT, "include"),
                        "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(exe)


@pytest.mark.parametrize("lo, hi", [(-4, 4), (-40, -4), (-125, -40), (4, 60), (60, 120)])
def test_relative_errors(program, lo, hi):
    r = subprocess.run([program, str(lo), str(hi)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    e1, e3 = (float(v) for v in r.stdout.split())
    assert e1 <= 1.001 * 2.0 ** -53
    assert e3 <= 1.01 * 2.0 ** -52
