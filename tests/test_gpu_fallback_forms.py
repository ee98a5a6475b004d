"""The forms that the far kernels fall back on, where a request has no polynomial form: the
tabulated FP32 form and the FP64 series, entry by entry against the oracle within the
parity bars (2e-5 and 1e-9 of max|Z|).  Cells several periods thick (the degrees grow with
the thickness) and cells of many orders; in the coarse thick cell near images lie
beyond the cut of the image series: their static part, which is integrated separately, has
to be taken out there too."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import cellgen
from oracle.fill import Problem, assemble
from oracle.topology import build_topology

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1809_05334_gb300", "csrc")

# nx, ny, nz, a, b, thickness; lambda, theta, phi; a near image beyond both cuts
CASES = [(2, 2, 2, 40.0, 40.0, 300.0, 500.0, 0.0, 0.0, True), (2, 2, 2, 40.0, 44.0, 300.0, 500.0, 0.5, 0.3, True),
         (2, 2, 12, 40.0, 40.0, 300.0, 500.0, 0.0, 0.0, False), (2, 2, 12, 44.0, 40.0, 300.0, 500.0, 0.6, 0.0, False),
         (2, 2, 12, 40.0, 40.0, 300.0, 500.0, 0.6, 0.4, False),
         (4, 4, 1, 700.0, 700.0, 100.0, 410.0, 0.0, 0.0, False), (4, 4, 1, 760.0, 760.0, 100.0, 410.0, 0.9, 0.7, False)]

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
    if (build_ewald_tables(a, b, k0, kx, ky, z, true, E, nullptr, &why)) return 1;
    Far64 f;
    std::vector<double> c64;
    build_far64(E, k0, kx, ky, f, c64);
    const double cut64 = (FP64_XCUT + 0.5) / E.E;
    if (build_ewald_tables(a, b, k0, kx, ky, z, false, E, nullptr, &why)) return 1;
    FarPoly p;
    std::vector<float> c;
    build_far_poly(E, make_ewald_f32(E), p, c);
    printf("%d %d %.17g %.17g\n", p.mode, f.n_blob, (FP32_XCUT + 0.5) / E.E, cut64);
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("forms")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "h.cpp"), os.path.join(CSRC, "ewald_tables.cpp"),
                    "-o", str(d / "h")], check=True)
    return str(d / "h")


def _cell(nx, ny, nz, a, b, d):
    return cellgen.slab_cell(nx, ny, nz, a, b, d, (3.9, 0.6), jitter=0.1 if nz > 2 else 0.0, seed=9)


@pytest.mark.parametrize("case", CASES)
def test_the_cells_take_the_fallback(harness, case):
    out = subprocess.run([harness] + [repr(v) for v in case[3:9]], check=True, capture_output=True, text=True).stdout.split()
    if case[3] < 100.0:
        assert int(out[1]) == 0          # the FP64 form (the wide cells may keep it)
    assert int(out[0]) == 0              # the FP32 form
    t = build_topology(_cell(*case[:6]))
    P = t["tet_verts"]
    cen = P.mean(axis=1)
    rho = np.max(np.linalg.norm(P - cen[:, None], axis=2), axis=1)
    reach = 0.0
    for m in (-1, 0, 1):
        for n in (-1, 0, 1):
            dist = np.linalg.norm(cen[:, None] - cen[None] + np.array([m * case[3], n * case[4], 0.0]), axis=2)
            near = dist < 1.5 * (rho[:, None] + rho[None])
            reach = max(reach, np.max(np.where(near, dist, 0.0)))
    assert (reach > float(out[3])) == case[9] and (reach > float(out[2])) >= case[9]


_ORACLE = {}


def _oracle(case):
    if case not in _ORACLE:
        cell = _cell(*case[:6])
        _ORACLE[case] = cell, assemble(Problem(build_topology(cell), *case[6:9], cell.eps(case[6])))
    return _ORACLE[case]


@pytest.mark.gpu
@pytest.mark.parametrize("case", CASES)
def test_fallback_matrix_fp64(case):
    vie = pytest.importorskip("paper_1809_05334_gb300.vie")
    cell, (Z, b) = _oracle(case)
    s = vie.Solver(precision=vie.VIE_FP64)
    try:
        s.set_mesh(cell)
        Z64, b64 = s.fill_matrix(*case[6:9], cell.eps(case[6]))
    finally:
        s.close()
    assert np.max(np.abs(Z64 - Z)) <= 1e-9 * np.max(np.abs(Z))
    assert np.max(np.abs(b64 - b)) <= 1e-9 * np.max(np.abs(b))


# The last cell is 1.85 wavelengths wide at oblique incidence: the splitting parameter is at
# its bound k0/6, where images and orders each carry a factor exp(9) that cancels between
# them, and FP32 keeps 8.7e-5 of max|Z| (both forms; the bar holds up to about exp(5)).
FP32_CASES = CASES[:-1] + [pytest.param(CASES[-1], marks=pytest.mark.xfail(strict=True, reason="exp(9) cancellation in FP32"))]


@pytest.mark.gpu
@pytest.mark.parametrize("case", FP32_CASES)
def test_fallback_matrix_fp32(case):
    vie = pytest.importorskip("paper_1809_05334_gb300.vie")
    cell, (Z, _) = _oracle(case)
    s = vie.Solver(precision=vie.VIE_FP32)
    try:
        s.set_mesh(cell)
        Z32 = s.fill_matrix_prec(*case[6:9], cell.eps(case[6]))
    finally:
        s.close()
    assert np.max(np.abs(Z32 - Z)) <= 2e-5 * np.max(np.abs(Z))
