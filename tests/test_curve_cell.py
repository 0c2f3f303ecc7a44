"""The curve's cells by multiplication (csrc/psum_internal.cuh, curve_cell) against the division that
defines them, floor((x / d + 1/2) 256) clamped to 0..255, on random positions, on both neighbours of
every cell face, on the box's faces and for positions outside the box or not finite (any cell in range).

Host only: compiled by the C++ compiler against the CUDA headers; skipped where either is missing."""
import os
import shutil
import subprocess

import pytest

from test_curve_key import CSRC, ROOT, _cuda_include

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <random>
#include "psum_internal.cuh"
static uint32_t by_division(double x, double d) {
    const int v = (int)std::floor((x / d + 0.5) * 256.0);
    return (uint32_t)(v < 0 ? 0 : v > 255 ? 255 : v);
}
int main(int argc, char** argv) {
    const double d = std::atof(argv[1]), inv = 256.0 / d;
    std::mt19937_64 rng(1);
    std::uniform_real_distribution<double> u(-0.5, 0.5);
    long bad = 0;
    auto check = [&](double x) {
        if (x >= -0.5 * d && x < 0.5 * d && psum::curve_cell(x, d, inv) != by_division(x, d)) ++bad;
    };
    for (int i = 0; i < 2000000; ++i) check(u(rng) * d);
    for (int c = 0; c <= 256; ++c)
        for (int k = -40; k <= 40; ++k) {
            const double f = (c / 256.0 - 0.5) * d;
            check(f);
            check(f + k * 1e-17 * d);
            check(f + k * 1e-9 * d);
            check(f + k * 2.5e-8 * d);
            double x = f;
            for (int s = 0; s < std::abs(k); ++s) x = std::nextafter(x, k < 0 ? -1e9 : 1e9);
            check(x);
        }
    const double wild[] = {d, -d, 1e300, -1e300, INFINITY, -INFINITY, NAN, 0.5 * d};
    for (double x : wild) bad += psum::curve_cell(x, d, inv) > 255;
    printf("%ld\n", bad);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = _cuda_include()
    if not cxx or not inc:
        pytest.skip("no host C++ compiler or CUDA headers")
    d = tmp_path_factory.mktemp("cell")
    src, exe = d / "cell.cpp", d / "cell"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-I", inc, "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(exe)


@pytest.mark.parametrize("d", ["1.0", "1.5", "2.0", "0.7310585786300049", "1e-3", "1024", "3e5"])
def test_cells_are_those_of_the_division(program, d):
    r = subprocess.run([program, d], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
    assert int(r.stdout) == 0
