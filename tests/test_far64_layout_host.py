"""Layout of the FP64 far form's table block (build_far64), built with the host compiler: the
kernels read a directory entry as one int4, so the directory starts on a 16-byte boundary
(an even number of doubles) whatever the number of images, and so does every entry."""
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
    const double a = atof(argv[1]), b = atof(argv[2]), th = atof(argv[3]), ph = atof(argv[4]), k0 = 6.283185307179586 / 500.0;
    const double kx = k0 * sin(th) * cos(ph), ky = k0 * sin(th) * sin(ph);
    static EwaldTables E;
    const char *why = "";
    if (build_ewald_tables(a, b, k0, kx, ky, 60.0, true, E, nullptr, &why)) return 1;
    Far64 f;
    std::vector<double> c;
    build_far64(E, k0, kx, ky, f, c);
    printf("%d %d %d %d %d\n", f.n_blob, f.n_img, f.img, f.dir, (int)c.size());
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("layout64")
    (d / "h.cpp").write_text(HARNESS)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "h.cpp"), os.path.join(CSRC, "ewald_tables.cpp"),
                    "-o", str(d / "h")], check=True)
    return str(d / "h")


@pytest.mark.parametrize("case", [(200.0, 200.0, 0.0, 0.0), (200.0, 120.0, 0.0, 0.0), (80.0, 80.0, 0.5, 0.0),
                                  (300.0, 150.0, 0.6, 0.3), (400.0, 90.0, 1.1, 0.8)])
def test_directory_on_a_16_byte_boundary(harness, case):
    out = subprocess.run([harness] + [repr(v) for v in case], check=True, capture_output=True, text=True).stdout
    n, n_img, img, at, size = (int(v) for v in out.split())
    assert n == size > 0 and at >= img + 4 * n_img
    assert at % 2 == 0
