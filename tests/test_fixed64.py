"""The float64 pair terms in 64-bit integer coordinates (csrc/fixed64.cuh), on the host, against long double:
differences with their largest in every binade that takes the integer form, small and zero ones beside it, both
signs, estimates up to three units in the last place off.  Bounds, in units of 2^-53 (half a unit in the last
place of 1..2): the rounding to 53 bits is one; the squared distance loses four units of 2^58 at the most
(2^-56), so 1/r another 2^-4 and q/r^3 another 3 2^-4 and 2^-4 for its integer products; the differences are
rounded once.  The conversion of coordinates is exact to half a unit and saturates.

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
#include "fixed64.cuh"
using namespace psum;
int main(int argc, char** argv) {
    const int top = std::atoi(argv[1]), k = std::atoi(argv[2]);
    std::mt19937_64 rng(7);
    const long double u = ldexpl(1.0L, -k);
    long double w1 = 0, w3 = 0, wd = 0, wc = 0;
    for (int it = 0; it < 300000; ++it) {
        FixedDelta d[3];
        for (int i = 0; i < 3; ++i) {
            long long v = 0;
            switch (rng() % 6) {
                case 0: v = (long long)(rng() >> (63 - rng() % (top + 1))); break;
                case 1: v = (1ll << top) - (long long)(rng() & 1); break;
                case 2: v = (1ll << (top + 1)) - 1 - (long long)(rng() & 1); break;
                case 3: v = (long long)(rng() & 1); break;
                default: v = (long long)(rng() >> (63 - top));
            }
            if (i == (int)(it % 3)) v |= 1ll << top;
            if (rng() & 1) v = -v;
            const long long t = (long long)(rng() >> 4) - (1ll << 59);
            d[i] = fixed_delta(t + v, t);
            const uint64_t a = d[i].a + (d[i].sign ? 1 : 0);
            if (a != (uint64_t)(v < 0 ? -v : v)) return 1;
        }
        const uint32_t high = (uint32_t)((d[0].a | d[1].a | d[2].a) >> 32);
        if (high < kFixedNear || high >= kFixedFar) continue;
        const FixedR2 r = fixed_r2(d[0], d[1], d[2], high);
        if (r.R < 1ull << 58 || r.R >= 1ull << 62) return 2;
        const long double X = d[0].a, Y = d[1].a, Z = d[2].a, rr = sqrtl(X * X + Y * Y + Z * Z) * u;
        const float y0 = (float)(1.0L / sqrtl((long double)fixed_estimate_arg(r.R)));
        for (int q = -3; q <= 3; ++q) {
            uint32_t yb;
            memcpy(&yb, &y0, 4);
            const FixedInverse v = fixed_inverse(r, k, yb + q);
            w1 = std::max(w1, fabsl(fixed_ri(v) * rr - 1));
            const double c = std::ldexp(1.0 + std::ldexp((double)(rng() >> 12), -52), (int)(rng() % 401) - 200) * (rng() & 1 ? 1 : -1);
            FixedCharge fc, f0;
            if (!fixed_charge(c, fc) || !fixed_charge(0.0, f0) || fixed_weight(fixed_cube(v), 3 * v.x, f0, 0.0) != 0) return 5;
            w3 = std::max(w3, fabsl(fixed_weight(fixed_cube(v), 3 * v.x, fc, c) * rr * rr * rr / c - 1));
        }
        for (int i = 0; i < 3; ++i) {
            const long double t = (d[i].sign ? -1.0L : 1.0L) * d[i].a * u, g = fixed_value(d[i], k);
            if (d[i].a) wd = std::max(wd, fabsl(g - t) / fabsl(t));
            else if (fabsl(g) > 0.25L * u) return 3;
        }
        const double c = std::ldexp((double)(long long)(rng() >> 1) * (rng() & 1 ? 1 : -1), top - 63 - k - (int)(rng() % 70));
        wc = std::max(wc, fabsl((long double)to_fixed(c, k) * u - c) / u);
    }
    FixedCharge no;
    const double big = std::ldexp(1.0, 62 - k);
    if (to_fixed(big, k) != kFixedOut || to_fixed(-4 * big, k) != kFixedOut || to_fixed(INFINITY, k) != kFixedOut ||
        to_fixed(-INFINITY, k) != kFixedOut || to_fixed(NAN, k) != kFixedOut || to_fixed(std::nextafter(big, 0.0), k) >= 1ll << 62 ||
        fixed_charge(4e-320, no) || fixed_charge(std::ldexp(1.0, 201), no) || fixed_charge(std::ldexp(-1.9, -201), no) ||
        to_fixed(0.0, k) || to_fixed(-5e-324, k) || to_fixed(1.0, kNoFixed) || to_fixed(-1e300, kNoFixed))
        return 4;
    for (long long t = -(1ll << 62) + 1; t < 1ll << 62; t += (1ll << 58) + 12345) {
        const FixedDelta d = fixed_delta(kFixedOut, t), b = fixed_delta(t, kFixedOut);
        if ((d.a >> 32) < kFixedFar || (b.a >> 32) < kFixedFar) return 6;
    }
    const long double h = ldexpl(1.0L, -53);
    printf("%Lg %Lg %Lg %Lg\n", w1 / h, w3 / h, wd / h, wc);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = _cuda_include()
    if not cxx or not inc:
        pytest.skip("no host C++ compiler or CUDA headers")
    d = tmp_path_factory.mktemp("fixed")
    src, exe = d / "fixed.cpp", d / "fixed"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", inc, "-I", os.path.join(ROOT, "include"),
                        "-I", CSRC, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(exe)


@pytest.mark.parametrize("top", [53, 54, 57, 60, 61])
@pytest.mark.parametrize("k", [2, 59, 122])
def test_relative_errors(program, top, k):
    r = subprocess.run([program, str(top), str(k)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    e1, e3, ed, ec = (float(v) for v in r.stdout.split())
    assert e1 <= 1.07
    assert e3 <= 1.26
    assert ed <= 1.0
    assert ec <= 0.5
