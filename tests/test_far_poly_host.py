"""Spectral polynomials of the far kernels (CPU, no GPU): build_far_poly
(csrc/ewald_tables.cpp) against the order sum with the orders' closed form.

The polynomials replace per-lane table entries, so every form they accept is
compared with the plain sum over the order rectangle: normal incidence, the
k_y = 0 fold and the full rectangle, square and unequal periods, thin cells
(degree 2) to cells several periods thick (the largest degrees), and the
refusal beyond.  Tolerance (derived): each coefficient is rounded to FP32
(2^-24 of it) and each column drops less than 1e-9 of the largest order, so
|error| <= sum_orders (2^-24 sum_n |c_n| + 1e-9 max|G|).
"""
import json
import os
import shutil
import subprocess

import numpy as np
import pytest
from scipy.special import wofz

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1809_05334_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "ewald_tables.h"
using namespace vie;
int main(int argc, char **argv) {
    const double a = atof(argv[1]), b = atof(argv[2]), lam = atof(argv[3]), th = atof(argv[4]), ph = atof(argv[5]);
    const double z = atof(argv[6]), k0 = 6.283185307179586 / lam;
    static EwaldTables E;
    const char *why = "";
    if (build_ewald_tables(a, b, k0, k0 * sin(th) * cos(ph), k0 * sin(th) * sin(ph), z, false, E, nullptr, &why)) return 1;
    static EwaldF32 F;
    F = make_ewald_f32(E);
    FarPoly p;
    std::vector<float> c;
    build_far_poly(E, F, p, c);
    printf("{\"mode\": %d, \"nq\": %d, \"rows\": %d, \"n\": %d, \"E\": %.17g, \"k0\": %.17g, \"Eih\": %.17g, \"ts\": %.17g,",
           p.mode, p.nq, p.rows, p.n_coef, E.E, k0, (double)F.Eih, (double)p.t_scale);
    printf("\"kx\": %.17g, \"ky\": %.17g, \"p0\": %d, \"np\": %d, \"q0\": %d, \"nqr\": %d, \"rect\": [",
           k0 * sin(th) * cos(ph), k0 * sin(th) * sin(ph), E.p0, E.np, E.q0, E.nq);
    for (int i = 0; i < E.np * E.nq; ++i) printf("%s%d", i ? "," : "", E.rect_tab[i]);
    printf("]");
    const int *v[4] = {p.off, p.deg, p.im_off, p.im_deg};
    const char *nm[4] = {"off", "deg", "im_off", "im_deg"};
    for (int k = 0; k < 4; ++k) {
        printf(", \"%s\": [", nm[k]);
        for (int i = 0; i < FP_ROWS; ++i) printf("%s%d", i ? "," : "", v[k][i]);
        printf("]");
    }
    printf(", \"c\": [");
    for (size_t i = 0; i < c.size(); ++i) printf("%s%.9g", i ? "," : "", c[i]);
    printf("]}\n");
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("farpoly")
    (d / "h.cpp").write_text(HARNESS)
    exe = d / "h"
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "h.cpp"), os.path.join(CSRC, "ewald_tables.cpp"),
                    "-o", str(exe)], check=True)
    return str(exe)


def _order(t, a, b, p, q, z):
    """G_pq(z) = [e^{gz} erfc(g/2E + zE) + e^{-gz} erfc(g/2E - zE)] / (4ab g)."""
    def erfc(u):
        v = np.where(u.real < 0, -u, u)
        r = wofz(1j * v) * np.exp(-v * v)
        return np.where(u.real < 0, 2 - r, r)
    E = t["E"]
    g = np.sqrt(complex((t["kx"] + 2 * np.pi * p / a) ** 2 + (t["ky"] + 2 * np.pi * q / b) ** 2 - t["k0"] ** 2))
    u = np.atleast_1d(np.asarray(z, complex))
    return (np.exp(g * u) * erfc(g / (2 * E) + u * E) + np.exp(-g * u) * erfc(g / (2 * E) - u * E)) / (4 * a * b * g)


# period a, b, lambda, theta, phi, thickness -> expected form (FarMode) and columns
CASES = [((200.0, 200.0, 500.0, 0.0, 0.0, 140.0), 1, 4), ((400.0, 400.0, 600.0, 0.0, 0.0, 160.0), 1, 5),
         ((150.0, 120.0, 430.0, 0.0, 0.0, 90.0), 1, None), ((40.0, 40.0, 400.0, 0.0, 0.0, 80.0), 1, 4),
         ((200.0, 200.0, 500.0, 0.0, 0.0, 0.5), 1, 4), ((60.0, 60.0, 500.0, 0.0, 0.0, 150.0), 1, 4),
         ((200.0, 200.0, 500.0, 0.5, 0.0, 140.0), 2, None), ((400.0, 400.0, 650.0, 0.9, 0.0, 160.0), 2, None),
         ((300.0, 240.0, 420.0, 1.2, 0.0, 60.0), 2, None), ((180.0, 150.0, 430.0, 0.6, 0.3, 100.0), 3, None),
         ((400.0, 400.0, 650.0, 0.9, 1.1, 160.0), 3, None), ((60.0, 54.0, 520.0, 0.35, 0.2, 60.0), 3, None)]


@pytest.mark.parametrize("case,mode,nq", CASES)
def test_polynomials_reproduce_the_order_sum(harness, case, mode, nq):
    out = subprocess.run([harness] + ["%r" % v for v in case], check=True, capture_output=True, text=True).stdout
    t = json.loads(out)
    a, b, _, _, _, zmax = case
    assert t["mode"] == mode and (nq is None or t["nq"] == nq), (t["mode"], t["nq"])
    c = np.array(t["c"])
    assert t["n"] == len(c) and t["Eih"] == 2.0 ** round(np.log2(t["Eih"]))
    ns = (t["nq"] + 1) // 2 * 2
    rng = np.random.default_rng(3)
    for z in [0.0, zmax] + list(rng.uniform(0, zmax, 6)):
        dx, dy = rng.uniform(-1, 1, 2) * np.array([a, b])
        tt = t["ts"] * (z * t["Eih"]) ** 2 - 1.0
        bound, gmax = 0.0, 0.0

        def poly(off, deg, j):
            nonlocal bound
            k = c[off + ns * np.arange(deg + 1) + j]          # highest power first
            bound += 2.0 ** -24 * np.abs(k).sum()
            return np.polyval(k, tt)
        S = T = 0j
        for i in range(t["rows"]):
            if mode == 1:
                X = 1.0 if i == 0 else 2 * np.cos(2 * np.pi * i / a * dx)
            else:
                X = np.exp(-1j * (t["kx"] + 2 * np.pi * (t["p0"] + i) / a) * dx)
            for j in range(t["nq"]):
                if mode == 3:
                    Y = np.exp(-1j * (t["ky"] + 2 * np.pi * (t["q0"] + j) / b) * dy)
                else:
                    Y = 1.0 if j == 0 else 2 * np.cos(2 * np.pi * j / b * dy)
                S += X * Y * poly(t["off"][i], t["deg"][i], j)
                if t["im_deg"][i] >= 0:
                    T += X * Y * poly(t["im_off"][i], t["im_deg"][i], j)
        ref, orders = 0j, 0
        for i in range(t["np"]):
            for j in range(t["nqr"]):
                if t["rect"][i * t["nqr"] + j] < 0:
                    continue
                p, q = t["p0"] + i, t["q0"] + j
                G = _order(t, a, b, p, q, z)[0]
                gmax = max(gmax, abs(_order(t, a, b, p, q, 0.0)[0]), abs(G))
                orders += 1
                ref += G * np.exp(-1j * ((t["kx"] + 2 * np.pi * p / a) * dx + (t["ky"] + 2 * np.pi * q / b) * dy))
        bound = 4 * bound + 2 * orders * 1e-9 * gmax + 1e-12 * orders * gmax   # weights up to 4; real and imaginary part
        assert abs(S + 1j * T - ref) <= bound, (case, z, abs(S + 1j * T - ref), bound)


def test_too_thick_a_cell_is_left_to_the_tabulated_form(harness):
    """Beyond E z_max ~ 7 an order needs more than the largest degree: no polynomial form."""
    out = subprocess.run([harness, "40", "40", "500", "0", "0", "300"], check=True, capture_output=True, text=True).stdout
    t = json.loads(out)
    assert t["mode"] == 0 and t["n"] == 0


HARNESS64 = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "ewald_tables.h"
using namespace vie;
int main(int argc, char **argv) {
    const double a = atof(argv[1]), b = atof(argv[2]), lam = atof(argv[3]), th = atof(argv[4]), ph = atof(argv[5]);
    const double z = atof(argv[6]), k0 = 6.283185307179586 / lam, kx = k0 * sin(th) * cos(ph), ky = k0 * sin(th) * sin(ph);
    static EwaldTables E;
    const char *why = "";
    if (build_ewald_tables(a, b, k0, kx, ky, z, true, E, nullptr, &why)) return 1;
    Far64 f;
    std::vector<double> c;
    build_far64(E, k0, kx, ky, f, c);
    printf("{\"n\": %d, \"sym\": %d, \"rows\": %d, \"cols\": %d, \"n_img\": %d, \"ts\": %.17g, \"kx0\": %.17g, \"ky0\": %.17g, "
           "\"xs\": %.17g, \"E\": %.17g, \"k0\": %.17g, \"bb\": %.17g, \"kx\": %.17g, \"ky\": %.17g, \"n_mode\": %d, \"dir\": [",
           f.n_blob, f.sym, f.rows, f.cols, f.n_img, f.t_scale, kx - f.i0 * f.sx, ky - f.j0 * f.sy, f.xs, E.E, k0, E.bb, kx, ky, E.n_mode);
    for (int i = 0; i < f.rows * f.cols; ++i) {
        int v[4];
        memcpy(v, &c[f.dir + 2 * i], sizeof(v));
        printf("%s[%d,%d,%d,%d]", i ? "," : "", v[0], v[1], v[2], v[3]);
    }
    printf("], \"c\": [");
    for (int i = 0; i < 2 * f.rows * f.cols; ++i) c[f.dir + i] = 0;   // ints, printed above
    for (int i = 0; i < f.n_blob; ++i) printf("%s%.17g", i ? "," : "", c[i]);
    printf("]}\n");
    return 0;
}
"""


@pytest.fixture(scope="module")
def harness64(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("far64")
    (d / "h.cpp").write_text(HARNESS64)
    exe = d / "h"
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "h.cpp"), os.path.join(CSRC, "ewald_tables.cpp"),
                    "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("case", [(200.0, 200.0, 500.0, 0.0, 0.0, 140.0), (150.0, 120.0, 430.0, 0.0, 0.0, 90.0),
                                  (40.0, 40.0, 400.0, 0.0, 0.0, 80.0), (200.0, 200.0, 500.0, 0.5, 0.0, 0.5),
                                  (180.0, 150.0, 430.0, 0.6, 0.3, 100.0), (400.0, 400.0, 650.0, 0.9, 1.1, 160.0)])
def test_fp64_form_reproduces_the_series(harness64, case):
    """The FP64 orders and spatial kernel against their closed forms: 2e-13 of the
    summed orders (the 40-term Faddeeva expansion behind the propagating orders and
    F carries 3e-14, Horner and the dropped terms a few 1e-16 each)."""
    out = subprocess.run([harness64] + ["%r" % v for v in case], check=True, capture_output=True, text=True).stdout
    t = json.loads(out)
    a, b, _, _, _, zmax = case
    assert t["n"] > 0 and t["sym"] == (case[3] == 0.0)
    c = np.array(t["c"])
    rng = np.random.default_rng(5)
    for z in [0.0, zmax] + list(rng.uniform(0, zmax, 4)):
        dx, dy = rng.uniform(-1, 1, 2) * np.array([a, b])
        tt = t["ts"] * z * z - 1.0
        g = ref = 0j
        size = 0.0
        for i in range(t["rows"]):
            for j in range(t["cols"]):
                ro, rd, io, idg = t["dir"][i * t["cols"] + j]
                G = 0j
                if rd >= 0:
                    G += np.polyval(c[ro:ro + rd + 1], tt)
                if idg >= 0:
                    G += 1j * np.polyval(c[io:io + idg + 1], tt)
                if t["sym"]:
                    w = (1 if i == 0 else 2 * np.cos(2 * np.pi * i / a * dx)) * (1 if j == 0 else 2 * np.cos(2 * np.pi * j / b * dy))
                    p, q = i, j
                else:
                    w = np.exp(-1j * ((t["kx0"] + 2 * np.pi * i / a) * dx + (t["ky0"] + 2 * np.pi * j / b) * dy))
                    p = i + int(round((t["kx0"] - t["kx"]) * a / (2 * np.pi)))
                    q = j + int(round((t["ky0"] - t["ky"]) * b / (2 * np.pi)))
                g += w * G
                if rd >= 0:
                    R = _order(t, a, b, p, q, z)[0]
                    ref += w * R
                    size += abs(w) * abs(_order(t, a, b, p, q, 0.0)[0])
        assert abs(g - ref) <= 2e-13 * size, (case, z, abs(g - ref) / size)
    # every order inside the cut is there
    kmax = 2.0 * t["E"] * 6.0 + t["k0"]
    n = sum(1 for p in range(-40, 41) for q in range(-40, 41)
            if np.hypot(t["kx"] + 2 * np.pi * p / a, t["ky"] + 2 * np.pi * q / b) <= kmax)
    have = sum((4 if i and j else 2 if i or j else 1) if t["sym"] else 1
               for i in range(t["rows"]) for j in range(t["cols"]) if t["dir"][i * t["cols"] + j][1] >= 0)
    assert have == n
    # spatial kernel F(x) = exp(-x^2) Re erfcx(x + j b)
    x = rng.uniform(0, 6.49, 400)
    u = x * t["xs"] / t["E"]
    i = u.astype(int)
    F = np.array([np.polyval(c[9 * k:9 * k + 9][::-1], v - k) for k, v in zip(i, u)])
    ref = np.exp(-x * x) * wofz(1j * (x + 1j * t["bb"])).real
    assert np.max(np.abs(F - ref)) <= 2e-13
