"""The far kernels leave the constant G_00(0) out of the charge term at normal incidence:
exact as long as no test function carries a net charge (checked on the host), and
what makes the FP32 matrix's imaginary part accurate.  There the imaginary part of
g_p is one order alone, without the images and the other orders of the real part,
so its error may not exceed the real part's (it was 1.6 times that)."""
import numpy as np
import pytest

import cellgen
from oracle.topology import KIND_HALF, build_topology

CELLS = {"cube": (lambda: cellgen.cube_cell(80.0, 20.0, 60.0, 40.0, 20.0), 560.0),
         "slab": (lambda: cellgen.slab_cell(4, 3, 2, 200.0, 160.0, 60.0, (3.9, 0.6), jitter=0.1, seed=9), 500.0),
         "tiny": (lambda: cellgen.small_cells()["plasmonic_tiny"], 520.0)}


@pytest.mark.parametrize("name", sorted(CELLS))
def test_test_functions_are_neutral(name):
    t = build_topology(CELLS[name][0]())
    q, area = np.zeros(t["n"]), np.zeros(t["n"])
    np.add.at(q, t["basis"].ravel(), (t["sign"] * t["area"]).ravel())
    np.maximum.at(area, t["basis"].ravel(), t["area"].ravel())
    cf = t["charge_faces"]
    half = cf[t["kind"][cf] == KIND_HALF]
    q[half] -= area[half]
    assert np.max(np.abs(q) / area) < 1e-13   # areas of matched faces, rounded in FP64


@pytest.mark.gpu
@pytest.mark.parametrize("name", sorted(CELLS))
def test_imaginary_part_of_the_matrix(name):
    vie = pytest.importorskip("paper_1809_05334_gb300.vie")
    cell, lam = CELLS[name][0](), CELLS[name][1]
    s = vie.Solver(precision=vie.VIE_FP32)
    try:
        s.set_mesh(cell)
        Z64, _ = s.fill_matrix(lam, 0.0, 0.0, cell.eps(lam))
        d = s.fill_matrix_prec(lam, 0.0, 0.0, cell.eps(lam)) - Z64
        assert np.max(np.abs(d)) <= 2e-5 * np.max(np.abs(Z64))
        assert np.sqrt(np.mean(d.imag ** 2)) <= np.sqrt(np.mean(d.real ** 2))
    finally:
        s.close()
