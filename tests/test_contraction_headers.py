"""The contraction's index arithmetic and weights as the kernels' headers have them, compiled
for the host: the constants that test_contraction_indexing.py copies, the rule that lets a
node take the contraction and the window weights it then uses (against the interpolation
they stand for), the staged slots every thread reads, and the shared memory of a block."""
import os
import shutil
import subprocess

import pytest

import test_contraction_indexing as copies

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
SRC = r"""
#include "pond_q27.cuh"
#include "pond_q16.cuh"
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>
using namespace pond;
static int bad = 0;
#define CHECK(c) do { if (!(c) && bad++ < 8) std::printf("line %d: %s\n", __LINE__, #c); } while (0)

// weights of one axis for the gauge (s, u): taken exactly when every floor is -1 or 0, and
// then, placed in the window of five nodes from -2 as the kernels place them, they interpolate
// cubic polynomials at the departure point
template <typename R, int Q, typename F>
void axis(const double (&c)[Q], R s, R u, R dt, double tol, F weights)
{
    R a[Q][4];
    bool near0[Q];
    const bool ok = weights(s, u, dt, a, near0);
    bool expect = true;
    for (int j = 0; j < Q; ++j) {
        const R d = -(s * (R)c[j] + u) * dt;
        const R f = std::floor(d);
        expect = expect && (f == R(0) || f == R(-1));
    }
    CHECK(ok == expect);
    if (!ok) return;
    for (int j = 0; j < Q; ++j) {
        const double d = (double)(-(s * (R)c[j] + u) * dt);
        for (int p = 0; p < 4; ++p) {
            double sum = 0.0;
            for (int k = 0; k < 4; ++k) sum += (double)a[j][k] * std::pow((double)((near0[j] ? 1 : 0) + k - HALO), p);
            CHECK(std::fabs(sum - std::pow(d, p)) <= tol);
        }
    }
}

template <typename R>
void weights(double tol)
{
    const double co = std::sqrt(3 + std::sqrt(6.0)), ci = std::sqrt(3 - std::sqrt(6.0));
    const double c9[3] = {-1, 0, 1}, c16[4] = {-co, -ci, ci, co};
    Lat16<R> L{};
    for (int k = 0; k < 4; ++k) L.c[k] = (R)c16[k];
    auto w9 = [](R s, R u, R dt, R (&a)[3][4], bool (&n)[3]) { return axis_weights<R>(s, u, dt, a, n); };
    auto w16 = [&](R s, R u, R dt, R (&a)[4][4], bool (&n)[4]) { return axis_weights16<R>(L, s, u, dt, a, n); };
    const R inf = std::numeric_limits<R>::infinity(), nan = std::numeric_limits<R>::quiet_NaN();
    const R special[] = {R(0), R(1e-30), R(0.5), R(0.9999999), R(1), R(1.7), R(3), R(1e4), inf, -inf, nan, R(-0.5), R(-1)};
    std::mt19937 g(7);
    std::uniform_real_distribution<double> rs(0.01, 2.0), ru(-2.5, 2.5);
    for (R dt : {R(0.1), R(0.5), R(1), inf}) {
        for (R s : special)
            for (R u : special) {
                axis<R, 3>(c9, s, u, dt, tol, w9);
                axis<R, 4>(c16, s, u, dt, tol, w16);
            }
        for (int k = 0; k < 4000; ++k) {
            axis<R, 3>(c9, (R)rs(g), (R)ru(g), dt, tol, w9);
            axis<R, 4>(c16, (R)rs(g), (R)ru(g), dt, tol, w16);
        }
    }
}

int main()
{
    std::printf("%d %d %d %d %d %d %d %d %d %d %d\n", HALO, STEP_NB, SPLIT_NB, AUXW, KQW, KEEP, SL, Slot<float>::stride,
                Slot<double>::stride, Slot16<float>::stride, Slot16<double>::stride);
    std::printf("%d %d %d %d %d %d\n", S27X * S27Y, PZ27, SLOT_SPACE27, Slot27<float>::stride, Slot27<double>::stride, K27_N);
    weights<double>(1e-13);
    weights<float>(4e-6);
    // D3Q27: the slots a thread's window reaches, and where the staged nodes lie
    for (int tid = 0; tid < Q27_THREADS; ++tid) {
        const int tx = tid % T27X, tz = (tid / T27X) % T27Z, ty = tid / (T27X * T27Z);
        const int own = (tz + HALO27) * PZ27 + (ty + HALO27) * PY27 + tx + HALO27, reach = 2 * (PZ27 + PY27 + 1);
        CHECK(ty < T27Y && own - reach >= 0 && own + reach < SLOT_SPACE27);
        CHECK(own == slot27(((tz + HALO27) * S27Y + ty + HALO27) * S27X + tx + HALO27));
    }
    for (int k = 0; k < SLOTS27; ++k) CHECK(slot27(k) >= 0 && slot27(k) < SLOT_SPACE27 && (k == 0 || slot27(k) > slot27(k - 1)));
    CHECK(2 * (q27_smem_bytes<float>() + 2048) <= 228 * 1024 && q27_smem_bytes<double>() + 2048 <= 227 * 1024);
    for (int tx = 1; tx <= STEP_NB; tx *= 2) {
        CHECK(q16_smem_bytes<float>(tx, STEP_NB / tx) + 2048 <= 227 * 1024);
        CHECK(q16_smem_bytes<double>(tx, STEP_NB / tx) + 2048 <= 227 * 1024);
    }
    return bad ? 1 : 0;
}
"""


def test_headers(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "contraction.cu", tmp_path / "contraction"
    src.write_text(SRC)
    subprocess.check_call([NVCC, "-std=c++17", "-O1", "-gencode=arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "paper_2002_09217_gb300", "csrc"), "-o", str(exe), str(src)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout
    first, second = [tuple(map(int, x.split())) for x in r.stdout.strip().split("\n")]
    assert first[:7] == (copies.HALO, copies.NB, copies.SPLIT, copies.AUX, copies.KQ, copies.KEEP, copies.SL)
    assert first[7:] == (20, 19, 36, 33)                   # slot strides of D2Q9 and D2Q16
    assert second == (12 * 8, 12 * 8 + 8, 8 * (12 * 8 + 8), 30, 27, 24)
