"""Masks of the warp shuffles: named in the source, never taken from the lanes that happen to run together
(__activemask says nothing of the others, which may be on their way).  The pair kernels join four neighbouring
threads, a target group each, under quad_mask: each of the four has the same mask and is in it, and a loop over
(image, group) entries by 128 threads takes all four of a quad through every trip or none, whatever images it spans.

Host only: compiled by the C++ compiler against the CUDA headers; skipped where either is missing."""
import glob
import os
import re
import shutil
import subprocess

import pytest

from test_curve_key import CSRC, ROOT, _cuda_include

PROGRAM = r"""
#include "psum_internal.cuh"
using namespace psum;
int main() {
    static_assert(kTgt32 == 4, "a quad per image");
    for (int t = 0; t < kThreads32; ++t) {
        const unsigned m = quad_mask(t);
        unsigned want = 0;
        for (int k = 0; k < 32; ++k)
            if (k / 4 == (t % 32) / 4) want |= 1u << k;
        if (m != want || !(m >> (t % 32) & 1u)) return 1;
    }
    for (int lo = 0; lo < 40; ++lo)
        for (int hi = lo; hi < lo + 100; ++hi)
            for (int t = 0; t < kThreads32; t += 4)
                for (int trip = 0; trip < 5; ++trip) {
                    int in = 0;
                    for (int k = 0; k < 4; ++k) in += lo * kTgt32 + t + k + trip * kThreads32 < hi * kTgt32;
                    if (in != 0 && in != 4) return 2;
                }
    return 0;
}
"""


def test_no_mask_is_taken_from_the_running_lanes():
    files = glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    assert files
    for f in files:
        with open(f) as h:
            assert not re.search(r"__activemask\s*\(", h.read()), f


def test_quads(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = _cuda_include()
    if not cxx or not inc:
        pytest.skip("no host C++ compiler or CUDA headers")
    src, exe = tmp_path / "quads.cpp", tmp_path / "quads"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-O2", "-std=c++17", "-I", inc, "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                        str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    assert subprocess.run([str(exe)], timeout=60).returncode == 0
