"""The grouped block preconditioner and the two-column GMRES at the block sizes where the
grouping changes (one group below 3,072 unknowns, two up to 6,143, four above).  A cell
of one domain has one block, the whole matrix, so the preconditioner is its inverse up to
the FP16 copies: every iteration then reduces the residual by at least 1e-1 (FP16 carries
5e-4 of each entry), so the 1e-8 asked for takes at most 8 iterations and a sweep's slack.
At normal incidence TE and TM converge together; at theta = 0.5 one comes first, which
leaves a right-hand side that is already solved in the block."""
import numpy as np
import pytest

import cellgen

pytestmark = pytest.mark.gpu

vie = pytest.importorskip("paper_1809_05334_gb300.vie")


@pytest.mark.parametrize("prec", ["FP32", "FP16"])
@pytest.mark.parametrize("n,theta", [(10, 0.0), (11, 0.5), (14, 0.0), (16, 0.5)])
def test_whole_matrix_block(n, theta, prec):
    cell = cellgen.slab_cell(n, n, 2, 200.0, 200.0, 40.0, (4.0, 0.5), jitter=0.1, seed=n)
    s = vie.Solver(precision=getattr(vie, "VIE_" + prec), tol=1e-8)
    try:
        size = s.set_mesh(cell)
        lo, hi = {10: (0, 3072), 11: (3072, 6144), 14: (3072, 6144), 16: (6144, 12000)}[n]
        assert lo <= size < hi
        r = s.solve(500.0, theta, 0.0, cell.eps(500.0), coeffs=True)
        assert r["status"] == 0 and np.max(r["rel_residual"]) <= 1e-8
        assert max(r["iterations"]) <= 12
        assert np.all(np.isfinite(r["x"]))
    finally:
        s.close()
