"""The pack kernel's integer chain (csrc/diffuse.cuh) against the recurrence that it restates,
v = fl32(q - carry), carry += v - q in float64: wherever the chain's own check holds for a whole
group, every float32 charge is the recurrence's; groups that it must refuse, it refuses.

Host only: compiled by the C++ compiler against the CUDA headers; skipped where either is missing."""
import os
import shutil
import subprocess

import pytest

from test_curve_key import CSRC, ROOT, _cuda_include

PROGRAM = r"""
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cmath>
#include <cstring>
#include <random>
#include <vector>
#include <cuda_runtime.h>
#include "diffuse.cuh"
using namespace psum;
static long long bits(double v) { long long b; memcpy(&b, &v, 8); return b; }
// 1: taken and equal, 0: refused, -1: taken and different
static int group(const std::vector<double>& q) {
    const int n = (int)q.size();
    int emax = 0;
    for (double v : q) emax = std::max(emax, exp_field(bits(v)));
    if (emax < kExpLo || emax > kExpHi) return 0;
    long long c = 0;
    std::vector<float> v(n);
    bool fine = true;
    for (int i = 0; i < n; ++i) {
        const long long Q = fixed_charge(bits(q[i]), emax), m = (1ll << dropped_bits(Q)) - 1;
        bool f;
        v[i] = (float)((double)diffuse_value(Q, c, f) * fixed_unit(emax));
        fine = fine && f;
        c = diffuse_step(Q + ((m + 1) >> 1), m, c);
    }
    if (!fine) return 0;
    double carry = 0.0;
    for (int i = 0; i < n; ++i) {
        const float r = (float)(q[i] - carry);
        carry += (double)r - q[i];
        if (r != v[i]) return -1;
    }
    return 1;
}
int main(int argc, char** argv) {
    const std::string kind = argv[1];
    std::mt19937_64 rng(5);
    std::normal_distribution<double> g;
    std::uniform_real_distribution<double> u(0.0, 1.0);
    int taken = 0, refused = 0, wrong = 0;
    for (int t = 0; t < 4000; ++t) {
        const int n = t % 3 == 0 ? 128 : 1 + (int)(u(rng) * 127);
        std::vector<double> q(n);
        for (int i = 0; i < n; ++i) {
            if (kind == "gauss") q[i] = g(rng);
            if (kind == "point8") q[i] = u(rng) < 0.5 ? 0.8 : -0.8;
            if (kind == "spread") q[i] = g(rng) * std::ldexp(1.0, -(int)(u(rng) * 12));
            if (kind == "zeros") q[i] = i && u(rng) < 0.3 ? 0.0 : 0.1 + g(rng);
            if (kind == "ties") q[i] = 1.0 + std::ldexp(1.0, -24);
            if (kind == "binade") q[i] = (i & 1 ? -1.0 : 1.0) * (i % 3 ? 0.7 : std::nextafter(1.0, 0.0));
            if (kind == "tiny") q[i] = g(rng) * 1e-30;
            if (kind == "huge") q[i] = g(rng) * 1e38;
            if (kind == "nan") q[i] = i == n / 2 ? NAN : g(rng);
        }
        const int r = group(q);
        taken += r == 1; refused += r == 0; wrong += r == -1;
    }
    printf("%d %d %d\n", taken, refused, wrong);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = _cuda_include()
    if not cxx or not inc:
        pytest.skip("no host C++ compiler or CUDA headers")
    d = tmp_path_factory.mktemp("diffuse")
    src, exe = d / "diffuse.cpp", d / "diffuse"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", inc, "-I", os.path.join(ROOT, "include"),
                        "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(exe)


# the least and the most share of groups that the chain takes
@pytest.mark.parametrize("kind, least, most", [("gauss", 0.99, 1.0), ("point8", 0.99, 1.0), ("spread", 0.9, 1.0),
                                               ("zeros", 0.0, 0.5), ("ties", 0.0, 0.0), ("binade", 0.0, 1.0),
                                               ("tiny", 0.0, 0.0), ("huge", 0.0, 1.0), ("nan", 0.0, 0.0)])
def test_chain_equals_the_float64_recurrence(program, kind, least, most):
    r = subprocess.run([program, kind], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
    taken, refused, wrong = (int(v) for v in r.stdout.split())
    assert wrong == 0
    assert least <= taken / (taken + refused) <= most
