"""Spacing of the spatial table, built with the host compiler: a power of two of the
distance for the far kernels, whose interval is then exact, and as fine as the table's
size allows for the allocation-free Green's function, whose FP32 results leave in
FP64 and are compared bit for bit from one version to the next."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1809_05334_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "ewald_tables.h"
using namespace vie;
int main(int argc, char **argv) {
    const double a = atof(argv[1]), b = atof(argv[2]), lam = atof(argv[3]), th = atof(argv[4]), k0 = 6.283185307179586 / lam;
    static EwaldTables E;
    const char *why = "";
    for (int pow2 = 0; pow2 < 2; ++pow2) {
        if (build_ewald_tables(a, b, k0, k0 * sin(th), 0.0, 60.0, false, E, nullptr, &why, 0.0, pow2)) return 1;
        const EwaldF32 F = make_ewald_f32(E, pow2);
        printf("%.17g %.17g %.17g %.17g %.17g\n", E.xs_h, (double)E.xs_max, E.E, (double)F.Eih, (double)(E.Ef * E.xs_inv_h));
    }
    printf("%d\n", NSPAT);
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("spacing")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "h.cpp"), os.path.join(CSRC, "ewald_tables.cpp"),
                    "-o", str(d / "h")], check=True)
    return str(d / "h")


@pytest.mark.parametrize("case", [(180.0, 150.0, 520.0, 0.35), (200.0, 200.0, 500.0, 0.0), (60.0, 54.0, 450.0, 0.0),
                                  (400.0, 400.0, 700.0, 1.2)])
def test_spacing(harness, case):
    out = subprocess.run([harness] + [repr(v) for v in case], check=True, capture_output=True, text=True).stdout.split("\n")
    (h, xm, _, eih, prod), (h2, xm2, e2, eih2, _) = ([float(v) for v in l.split()] for l in out[:2])
    n = int(out[2])
    assert h == xm / n and eih == prod                        # the finest, nothing rounded to a power of two
    m = eih2
    while m > 1.0:
        m /= 2.0
    while m < 1.0:
        m *= 2.0
    assert m == 1.0 and abs(h2 * eih2 / e2 - 1.0) < 1e-15     # index and nodes at the same distances
    assert xm2 <= n * h2 < 2.0001 * xm2                       # the cut in the table's upper half
