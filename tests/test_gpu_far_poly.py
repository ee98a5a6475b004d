"""The polynomial form of the FP32 far kernels on the GPU, at the sizes where its
pieces change: every column count of the three forms, thin and thick cells
(lowest and highest degrees), unequal periods, the step over to the tabulated
form, element counts around the 128-thread blocks.  FP32 Z and g_p against
the library's own FP64 series (itself checked against the oracle to 1e-9),
within the FP32 bars of the parity tests: 2e-5 max|Z|, 2e-6 max|g|."""
import numpy as np
import pytest

import cellgen

pytestmark = pytest.mark.gpu

vie = pytest.importorskip("paper_1809_05334_gb300.vie")

# slab cells: nx, ny, nz, a, b, thickness, lambda, theta, phi
CASES = [(3, 3, 1, 200.0, 200.0, 140.0, 500.0, 0.0, 0.0),      # normal, four columns
         (4, 4, 2, 400.0, 400.0, 160.0, 600.0, 0.0, 0.0),      # five columns
         (3, 2, 2, 150.0, 120.0, 30.0, 430.0, 0.0, 0.0),       # unequal periods
         (4, 4, 3, 60.0, 60.0, 120.0, 500.0, 0.0, 0.0),        # high degree
         (3, 3, 1, 200.0, 200.0, 1.0, 500.0, 0.0, 0.0),        # lowest degrees
         (4, 4, 2, 200.0, 200.0, 100.0, 500.0, 0.5, 0.0),      # fold
         (4, 3, 2, 300.0, 240.0, 60.0, 420.0, 1.2, 0.0),
         (4, 4, 2, 400.0, 400.0, 160.0, 650.0, 0.9, 0.0),
         (3, 3, 2, 180.0, 150.0, 100.0, 430.0, 0.6, 0.3),      # full rectangle
         (4, 4, 2, 400.0, 400.0, 160.0, 650.0, 0.9, 1.1),
         (2, 2, 1, 60.0, 54.0, 20.0, 520.0, 0.35, 0.2)]


@pytest.mark.parametrize("nx,ny,nz,a,b,d,lam,th,ph", CASES)
def test_fp32_fill_and_green(nx, ny, nz, a, b, d, lam, th, ph):
    cell = cellgen.slab_cell(nx, ny, nz, a, b, d, (3.9, 0.6), jitter=0.1 if min(nx, ny, nz) > 1 else 0.0, seed=9)
    s = vie.Solver(precision=vie.VIE_FP32)
    try:
        s.set_mesh(cell)
        eps = cell.eps(lam)
        Z64, _ = s.fill_matrix(lam, th, ph, eps)
        Z32 = s.fill_matrix_prec(lam, th, ph, eps)
        assert np.max(np.abs(Z32 - Z64)) <= 2e-5 * np.max(np.abs(Z64))
        p = np.random.default_rng(2).uniform(-0.99, 0.99, (1001, 3)) * np.array([a, b, d])
        g64 = s.green(p, lam, th, ph, vie.VIE_FP64)
        g32 = s.green(p, lam, th, ph, vie.VIE_FP32)
        assert np.max(np.abs(g32 - g64)) <= 2e-6 * np.max(np.abs(g64))
    finally:
        s.close()
