"""The Kannala-Brandt angles' bounded searches (csrc/kb_angles.h) against the plain walk
over the grid: the same doubles for gentle, wild, zero, NaN and infinite coefficients."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_24053_gb300", "csrc")

PROGRAM = r"""
#include "kb_angles.h"
#include <cstdio>
#include <random>
using namespace geer;
static double walk_fov_y(const float k[4], double fx, double w, double h) {
    const double edge = kb_theta_d(k, 0.5 * fx);
    if (!(edge > 0.0)) return NAN;
    const double target = edge * h / w;
    double lo = 0.0, hi = 0.5 * fx;
    for (int s = 1; s <= 8192; ++s) {
        const double ph = 0.5 * fx * s / 8192;
        if (kb_theta_d(k, ph) >= target) { hi = ph; lo = 0.5 * fx * (s - 1) / 8192; break; }
    }
    for (int it = 0; it < 200; ++it) {
        const double mid = 0.5 * (lo + hi);
        if (kb_theta_d(k, mid) >= target) hi = mid; else lo = mid;
    }
    return 2.0 * hi;
}
static double walk_phi_max(const float k[4]) {
    double prev = 0.0;
    for (int s = 1; s <= 4096; ++s) {
        const double val = kb_theta_d(k, M_PI * s / 4096);
        if (!(val > prev)) return M_PI * (s - 1) / 4096;
        prev = val;
    }
    return M_PI;
}
static bool same(double a, double b) { return a == b || (a != a && b != b); }
int main() {
    std::mt19937 rng(1);
    std::uniform_real_distribution<double> u(0, 1);
    std::normal_distribution<double> g;
    int bad = 0, turns = 0, ups = 0;
    for (int i = 0; i < 4000; ++i) {
        const double scale = i % 7 ? std::pow(10.0, -3.0 + 3.0 * u(rng)) : 0.0;
        float k[4];
        for (int j = 0; j < 4; ++j) k[j] = (float)(g(rng) * scale * std::pow(0.2, j));
        if (i % 50 == 0) k[i / 50 % 4] = i % 100 ? NAN : INFINITY;
        const float fx = (float)(0.02 + 6.2 * u(rng));
        const int w = 1 + (int)(2000 * u(rng)), h = 1 + (int)(2000 * u(rng));
        bad += !same(walk_fov_y(k, fx, w, h), kb_fov_y(k, fx, w, h));
        bad += !same(walk_phi_max(k), kb_phi_max(k));
        turns += kb_phi_max(k) < M_PI;
        ups += kb_fov_y(k, fx, w, h) > 0.0;
    }
    std::printf("%d %d %d\n", bad, turns, ups);
    return bad != 0;
}
"""


def test_bounded_searches_give_the_walks_doubles(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "kb.cpp", tmp_path / "kb"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O3", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    bad, turns, ups = map(int, out.stdout.split())
    assert out.returncode == 0 and bad == 0
    assert turns > 500 and ups > 2000  # both outcomes of either search occur
