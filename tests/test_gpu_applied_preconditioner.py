"""The preconditioner as a solve applies it: blocks of one, two and four groups side by side
(below 3,072 unknowns, up to 6,143, above), none of a size or an offset that is a multiple of
128.  After one GMRES iteration from x = 0 each polarisation's currents are a multiple of
M^-1 b, so a solve stopped there gives M^-1 b itself, through the grouped factors, their FP16
copies with two scales, the steps that several blocks share and the reads past a block's last
chunk.  Against the FP64 inverse of every domain block, with the bar of the block inverse:
8 u cond_2, u = 2^-11 (and below one half); a wrong step, scale or offset is O(1)."""
import numpy as np
import pytest
import scipy.linalg as sla

import cellgen
from oracle.solve import unknown_domains
from oracle.topology import build_topology

pytestmark = pytest.mark.gpu

vie = pytest.importorskip("paper_1809_05334_gb300.vie")

U16 = 2.0 ** -11
LAM, THETA = 550.0, 0.4


def _norm2(apply, apply_h, n, steps=12):
    """2-norm of an operator by power iteration (from below, within a few per cent)."""
    v = np.random.default_rng(1).standard_normal(n) + 0j
    for _ in range(steps):
        v = apply_h(apply(v / np.linalg.norm(v)))
    return np.sqrt(np.linalg.norm(v))


@pytest.fixture(scope="module")
def problem():
    cell = cellgen.layered_cell(220.0, 240.0, [(20.0, "buffer"), (40.0, "active"), (80.0, "buffer")], h_coarse=20.0, h_z=20.0,
                                jitter=0.1, seed=5)
    topo = build_topology(cell)
    udom = unknown_domains(topo, cell.eps(LAM))
    s = vie.Solver(precision=vie.VIE_FP64)
    try:
        s.set_mesh(cell)
        Z, b = s.fill_matrix(LAM, THETA, 0.0, cell.eps(LAM))
    finally:
        s.close()
    blocks = []
    for d in range(cell.n_domains):
        idx = np.nonzero(udom == d)[0]
        A = Z[np.ix_(idx, idx)]
        lu = sla.lu_factor(A)
        inv = _norm2(lambda v: sla.lu_solve(lu, v), lambda v: sla.lu_solve(lu, v, trans=2), len(idx))
        blocks.append((idx, sla.lu_solve(lu, b[idx]), inv * _norm2(lambda v: A @ v, lambda v: A.conj().T @ v, len(idx))))
    return cell, blocks


@pytest.mark.parametrize("prec,pivot", [("FP32", 512), ("FP32", 1024), ("FP16", 512), ("FP64", 512)])
def test_one_iteration_applies_the_block_inverses(problem, prec, pivot):
    cell, blocks = problem
    sizes = [len(i) for i, _, _ in blocks]
    assert sizes[0] < 3072 <= sizes[1] < 6144 <= sizes[2] and all(n % 128 for n in sizes) and all(np.cumsum(sizes)[:2] % 128)
    s = vie.Solver(precision=getattr(vie, "VIE_" + prec), tol=1e-6, max_iter=1, precond_pivot=pivot)
    try:
        s.set_mesh(cell)
        r = s.solve(LAM, THETA, 0.0, cell.eps(LAM), coeffs=True)
    finally:
        s.close()
    assert r["status"] == 1 and list(r["iterations"]) == [1, 1]
    for p in range(2):
        # the multiple from the whole vector, then block by block
        z = np.concatenate([v[:, p] for _, v, _ in blocks])
        x = np.concatenate([r["x"][i, p] for i, _, _ in blocks])
        c = np.vdot(z, x) / np.vdot(z, z)
        for i, v, cond in blocks:
            assert np.linalg.norm(r["x"][i, p] / c - v[:, p]) <= min(8 * U16 * cond, 0.5) * np.linalg.norm(v[:, p]), (len(i), cond)
