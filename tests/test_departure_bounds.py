"""Stencil nodes of a departure point stay on the grid whatever the gauge: the D2Q16 and
D3Q27 per-pair streams' index functions, compiled for the host from the kernels' headers
under the undefined-behaviour sanitizer (signed overflow, float to int out of range), over
NaN, infinite, huge and ordinary velocities at the grid's edges, both precisions and both
boundary rules."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

SRC = r"""
#include "pond_q27.cuh"
#include "pond_q16.cuh"
#include <cmath>
#include <cstdio>
#include <limits>
using namespace pond;

template <typename R>
int check(const char *name)
{
    const R inf = std::numeric_limits<R>::infinity(), big = std::numeric_limits<R>::max();
    const R v[] = {std::numeric_limits<R>::quiet_NaN(), inf, -inf, big, -big, R(3e9), R(-3e9), R(2147483648.0),
                   R(-2147483648.0), R(1e6), R(-1e6), R(2.5), R(-2.5), R(0)};
    int bad = 0;
    for (R x : v)
        for (int n : {1, 2, 48, 600000})
            for (int X : {0, 1, n / 2, n - 1})
                for (int bc : {0, 1}) {
                    if (X < 0 || X >= n) continue;
                    R w[4];
                    const int s[2] = {departure<R>(X, x, R(1), w), depart<R>(X, x, R(1), w)};
                    for (int f = 0; f < 2; ++f)
                        for (int k = 0; k < 4; ++k) {
                            const int i = bc_wrap(s[f] + k, n, bc);
                            if (i < 0 || i >= n) {
                                if (bad++ < 5) std::printf("%s v=%g n=%d X=%d bc=%d -> %d\n", name, (double)x, n, X, bc, i);
                            }
                            // ordinary velocities: the floor of the departure point less one
                            if (std::fabs((double)x) < 1e7 && s[f] != X + (int)std::floor(-(double)x) - 1) {
                                if (bad++ < 5) std::printf("%s v=%g n=%d X=%d starts at %d\n", name, (double)x, n, X, s[f]);
                            }
                        }
                }
    return bad;
}

int main() { return check<float>("float") + check<double>("double") ? 1 : 0; }
"""


def test_departure_stencils_stay_on_the_grid(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "departure.cu", tmp_path / "departure"
    src.write_text(SRC)
    subprocess.check_call([NVCC, "-std=c++17", "-O1", "-gencode=arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "paper_2002_09217_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                           "-Xcompiler", "-fsanitize=undefined", "-Xcompiler", "-fsanitize=float-cast-overflow",
                           "-Xcompiler", "-fno-sanitize-recover=all", "-o", str(exe), str(src), "-lubsan"])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
