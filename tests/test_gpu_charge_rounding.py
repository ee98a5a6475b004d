"""Rounding of the far entries of the FP32 matrix at oblique incidence.  An entry is the sum of
four element pairs' charge terms, each of the size v = A_m A_n |kappa g_p|, which cancel
almost entirely.  Each is rounded once on its way into Z (0.42 u rms of it, u = 2^-24) and
three of the four additions round a partial sum of up to 1.2 v: 1.2 u v together, 0.6 u of
|(v_1 .. v_4)| = 2 v.  The 16 values of a pair carry up to 4 u rms each, averaged by their
sum: 1 u of it.  Together 1.2; the bar is 1.3 u (with every factor rounded on the way it was
1.64 to 1.72, in the per-lane form before 1.95 to 2.08)."""
import numpy as np
import pytest

import cellgen
from oracle.topology import KIND_HALF, build_topology

pytestmark = pytest.mark.gpu

vie = pytest.importorskip("paper_1809_05334_gb300.vie")

CASES = [(5, 5, 3, 200.0, 180.0, 120.0, 500.0, 0.5, 0.0), (5, 4, 3, 180.0, 150.0, 100.0, 430.0, 0.6, 0.3),
         (5, 5, 3, 300.0, 240.0, 120.0, 650.0, 1.2, 0.0)]


@pytest.mark.parametrize("nx,ny,nz,a,b,d,lam,th,ph", CASES)
def test_far_entries(nx, ny, nz, a, b, d, lam, th, ph):
    cell = cellgen.slab_cell(nx, ny, nz, a, b, d, (3.9, 0.6), jitter=0.1, seed=9)
    eps = cell.eps(lam)
    t = build_topology(cell)
    P = t["tet_verts"]
    cen = P.mean(axis=1)
    rho = np.max(np.linalg.norm(P - cen[:, None], axis=2), axis=1)
    nt = len(cen)
    diff = (cen[:, None] - cen[None]).reshape(-1, 3)
    far = np.ones((nt, nt), bool)
    for m in (-1, 0, 1):
        for n in (-1, 0, 1):
            dist = np.linalg.norm(diff + np.array([m * a, n * b, 0.0]), axis=1).reshape(nt, nt)
            far &= dist > 1.5 * (rho[:, None] + rho[None])
    diff[np.all(diff == 0, axis=1)] = 1.0                      # the element itself: not far
    s32, s64 = vie.Solver(precision=vie.VIE_FP32), vie.Solver(precision=vie.VIE_FP64)
    try:
        s32.set_mesh(cell)
        s64.set_mesh(cell)
        g = np.abs(s64.green(diff, lam, th, ph, vie.VIE_FP64)).reshape(nt, nt)
        dZ = s32.fill_matrix_prec(lam, th, ph, eps) - s64.fill_matrix(lam, th, ph, eps)[0]
    finally:
        s32.close()
        s64.close()
    # functions on two tetrahedra of the cell itself
    k = np.nonzero((t["kind"] != KIND_HALF) & ~np.any(t["shift"][t["tm"], t["im"]] != 0, axis=-1))[0]
    tp, tm, area = t["tp"][k], t["tm"][k], t["area"][t["tp"][k], t["ip"][k]]
    kappa = abs(1.0 - 1.0 / np.conj(eps[0]))
    pairs = [np.ix_(x, y) for x in (tp, tm) for y in (tp, tm)]
    size = np.sqrt(sum((area[:, None] * area[None] * kappa * g[i]) ** 2 for i in pairs))
    ok = np.all([far[i] for i in pairs], axis=0)
    assert ok.sum() > 1000
    err = np.sqrt(np.mean((np.abs(dZ[np.ix_(k, k)]) / size)[ok] ** 2))
    assert err <= 1.3 * 2.0 ** -24, err * 2.0 ** 24
