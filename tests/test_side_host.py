"""The side a neighbour lies on, read from split float positions
(csrc/lp_split.h, side_of_split), against the sign of the FP64 offset with its
minimum image: open and periodic axes, boxes at and away from the origin,
offsets around 0, L/4, L/2, 3L/4 and L.  Compiled with the host C++ compiler;
needs no GPU."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
HEADER = os.path.join(HERE, "..", "paper_2206_11998_gb300", "csrc", "lp_split.h")

PROGRAM = r"""
#include "lp_split.h"
#include <cmath>
#include <cstdio>
#include <random>

static long n = 0, decided = 0, bad = 0;

static void check(bool per, double lo, double L, double xi, double xj)
{
    double d = xj - xi;
    if (per) { if (d > 0.5 * L) d -= L; else if (d < -0.5 * L) d += L; }
    const int want = d > 0 ? 1 : (d < 0 ? -1 : 0);
    const bool ok = std::fabs(lo) <= 0x1p20 * L && std::fabs(lo + L) <= 0x1p20 * L;
    const float near = ok ? 0.25f * (float)L : -1.0f;
    const float hi = (float)xi, li = (float)(xi - (double)hi), hj = (float)xj, lj = (float)(xj - (double)hj);
    const int got = lp::side_of_split(per, near, hi, li, hj, lj);
    ++n;
    if (got == lp::SIDE_FP64) return;
    ++decided;
    if (got != want) { if (bad < 5) printf("lo %a L %a xi %a xj %a: %d / %d\n", lo, L, xi, xj, got, want); ++bad; }
}

int main()
{
    std::mt19937_64 g(11);
    auto U = [&] { return (g() >> 11) * 0x1p-53; };
    const double los[] = {0.0, -0.5, 3.0, -1000.0, 1e6, 1e9}, Ls[] = {1.0, 0.37, 16.0, 1e-3};
    const double at[] = {0.0, 0.25, 0.5, 0.75, 1.0};
    for (double lo : los)
        for (double L : Ls)
            for (long t = 0; t < 60000; ++t) {
                const double xi = lo + L * U();
                double off = t % 3 == 0 ? L * (2 * U() - 1) : L * at[t % 5] + L * (U() - 0.5) * std::exp2(-(double)(g() % 50));
                if (g() & 1) off = -off;
                double xj = xi + off;
                if (xj < lo) xj += L; else if (xj >= lo + L) xj -= L;
                check(true, lo, L, xi, xj);
                check(false, lo, L, xi, xi + off);
            }
    check(true, 0.0, 1.0, 0.3, 0.3);
    check(true, 0.0, 1.0, 0.0, 1.0);
    printf("checked %ld decided %ld bad %ld\n", n, decided, bad);
    return bad != 0 || decided < n / 2;
}
"""


def test_side_of_split_matches_the_fp64_offset(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src = tmp_path / "side_check.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "side_check"
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.dirname(HEADER), str(src), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    print(r.stdout)
    assert r.returncode == 0, r.stdout
