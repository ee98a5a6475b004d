"""Where the GMRES of the mixed paths stops: TE and TM in one Krylov space each, as the
oracle's GMRES on the same FP32 matrix with exact block inverses.  The FP16 copies of the
inverses (5e-4 of an entry) move a residual that falls by about 0.7 an iteration by
less than one iteration, and the two iterates by less than the distance that one iteration
makes, 0.3 of the distance to the converged solution; a space over both polarisations
takes 20 to 35 % fewer iterations and stops somewhere else."""
import numpy as np
import pytest

import cellgen
from oracle.fill import Problem, rhs
from oracle.solve import block_preconditioner, gmres, solve_dense, unknown_domains
from oracle.topology import build_topology

pytestmark = pytest.mark.gpu

vie = pytest.importorskip("paper_1809_05334_gb300.vie")


@pytest.mark.parametrize("lam,theta,phi", [(520.0, 0.0, 0.0), (620.0, 0.6, 0.0), (560.0, 0.35, 0.4)])
def test_stops_where_separate_spaces_stop(lam, theta, phi):
    cell = cellgen.layered_cell(200.0, 200.0, [(40.0, "buffer"), (100.0, "active")], spheres=[(100.0, 100.0, 90.0, 20.0, "ag")],
                                h_coarse=40.0, h_fine=16.7, h_z=40.0, jitter=0.1, seed=3, lateral_fine=False)
    eps, tol = cell.eps(lam), 1e-4
    s = vie.Solver(precision=vie.VIE_FP32, tol=tol)
    try:
        s.set_mesh(cell)
        Z = s.fill_matrix_prec(lam, theta, phi, eps)
        r = s.solve(lam, theta, phi, eps, coeffs=True)
    finally:
        s.close()
    assert r["status"] == 0 and np.max(r["rel_residual"]) <= tol
    topo = build_topology(cell)
    b = rhs(Problem(topo, lam, theta, phi, eps))
    M, exact = block_preconditioner(Z, unknown_domains(topo, eps)), solve_dense(Z, b)
    for p in range(2):
        x, its, _ = gmres(Z, b[:, p], M, tol=tol)
        assert abs(r["iterations"][p] - its) <= 1
        assert np.linalg.norm(r["x"][:, p] - x) <= 0.7 * np.linalg.norm(x - exact[:, p])
