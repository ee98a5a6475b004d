"""FP64 solves as they are stopped.  At a tolerance of 1e-8 the iteration ends after three or four
steps, with currents some 1e-9 from the converged ones, and which ones they are follows from the
roundings of the preconditioner: FP32 inverses of the domain blocks by Gauss-Jordan with 128-wide
pivots inverted in registers, their products with FP16 operands, copied to FP16.  Results in double
precision hold to 1e-9 against recorded ones of that inverse (six unknowns of four slabs, both
polarisations; another inverse as good as this one moves them by up to 4e-9), and the iteration
counts are the recorded ones."""
import numpy as np
import pytest

import cellgen
from paper_1809_05334_gb300 import vie

pytestmark = pytest.mark.gpu

# slab_cell's n and m, wavelength, theta, phi, seed, iterations, currents of the unknowns linspace(0, N - 1, 6)
RECORDED = [
    (3, 1, 593.4032128981443, 0.23655668067532232, 0.4832568040755624, 19, (4, 4), [
        (complex(-1.134098022907e+00, 8.827947213336e-01), complex(2.139354991472e+00, -1.647019484289e+00)),
        (complex(5.826425577213e-01, -5.003522067677e-01), complex(-9.443294885090e-01, 7.897823352359e-01)),
        (complex(-1.058582482340e+00, 1.028660562503e+00), complex(-3.943431519713e-01, 4.208138137428e-01)),
        (complex(-9.641565658278e-03, -1.848573467256e-03), complex(3.010120113237e-01, 1.138729029603e-01)),
        (complex(-9.970926542926e-03, -3.199630275114e-03), complex(3.085455039992e-01, 9.009964200273e-02)),
        (complex(1.521730851525e-02, 3.913618876392e-02), complex(3.026925510103e-01, 3.128314937675e-02)),
    ]),
    (4, 1, 773.8291604179833, 0.0, 0.9195190814543128, 18, (3, 3), [
        (complex(-2.543941036830e+00, 1.087914205121e+00), complex(1.715333633130e+00, -7.758919757181e-01)),
        (complex(-1.121424322437e+00, 3.191610719868e-01), complex(-1.545418602732e+00, 4.849857184807e-01)),
        (complex(1.995135617912e+00, -6.426388598677e-01), complex(2.314720092123e+00, -7.139900097379e-01)),
        (complex(3.002546311804e+00, -8.760147293664e-01), complex(5.228857387910e-01, -1.547524722803e-01)),
        (complex(3.134133607688e-03, -4.728557962682e-03), complex(4.383077527480e-04, 4.834353903484e-02)),
        (complex(-7.862517580979e-04, -4.547393909846e-03), complex(-1.349958747344e-02, 5.044005876252e-02)),
    ]),
    (4, 1, 766.8419430717748, 0.0, 0.0, 4, (3, 3), [
        (complex(6.838447442682e-03, -1.948054877853e-02), complex(3.056570447844e+00, -1.335134200765e+00)),
        (complex(-1.900910548378e+00, 5.769644468683e-01), complex(1.385710855016e-01, -2.306517178794e-02)),
        (complex(3.043857255004e+00, -9.454375977763e-01), complex(7.056854500773e-02, -6.056407068665e-03)),
        (complex(2.233772195006e+00, -6.578360382476e-01), complex(-2.059414939217e+00, 6.017755648658e-01)),
        (complex(2.538978018257e-03, 3.422750555868e-02), complex(-2.363150742881e-03, 3.281069084831e-02)),
        (complex(-1.231736708793e-02, 4.319596621552e-02), complex(-8.379960692958e-03, 3.851922864289e-02)),
    ]),
    (5, 3, 629.8975322424188, 0.4405629616786337, 0.0, 14, (3, 3), [
        (complex(7.773264331024e-03, -2.718837015796e-02), complex(2.280041789231e+00, -2.029013921799e+00)),
        (complex(-4.265336900231e-03, 2.514704752578e-04), complex(-3.272605507224e-01, 1.632169516020e-01)),
        (complex(1.417950285937e+00, -1.740128448744e+00), complex(-1.453338186309e+00, 1.668951915965e+00)),
        (complex(1.090159757040e+00, -1.927693350824e+00), complex(-1.165755685276e+00, 1.914283657479e+00)),
        (complex(7.694504666235e-01, -2.141119118966e+00), complex(-8.049372480061e-01, 2.029622141086e+00)),
        (complex(5.434482111846e-03, 2.392616079777e-02), complex(5.221564358410e-01, -1.449041521682e-01)),
    ]),
]


@pytest.mark.parametrize("case", RECORDED, ids=["126", "224", "224b", "950"])
def test_stopped_solution_is_the_recorded_one(case):
    n, m, lam, theta, phi, seed, iterations, x = case
    cell = cellgen.slab_cell(n, n, m, 200., 200., 40., (4.0, .5), jitter=.1, seed=seed)
    s = vie.Solver(precision=vie.VIE_FP64, tol=1e-8)
    try:
        N = s.set_mesh(cell)
        r = s.solve(lam, theta, phi, cell.eps(lam), coeffs=True)
    finally:
        s.close()
    assert tuple(r["iterations"]) == iterations
    got = np.asarray(r["x"])[np.linspace(0, N - 1, 6).astype(int)]
    want = np.array(x)
    assert np.linalg.norm(got - want) <= 1e-9 * np.linalg.norm(want)
