"""The work that users of the solver have it do, as measurable cases.

A case names a unit cell, an incidence, a precision and the public entry point
it goes through; listed() holds one of each kind that is in use, from a handful
of Green's-function values to a 49k-unknown cell, and draw() gives more of the
same ranges.

kinds
  green   allocation-free periodic Green's function at device points
  solve   one (lambda, theta, phi) solve, TE and TM, on a mesh that is set
  remesh  a new mesh and its first solve (geometry scans, optimisation loops)
  batch   a wavelength x angle sweep of one mesh in concurrent solve slots
  serve   a solve server: requests of different meshes, submitted together
"""
import ctypes
import math

import numpy as np
import torch

import cellgen
from paper_1809_05334_gb300 import vie

PREC = {"fp64": vie.VIE_FP64, "fp32": vie.VIE_FP32, "fp16": vie.VIE_FP16, "bf16": vie.VIE_BF16}


def listed():
    return [
        # the smallest call: field probes of a framework that owns device memory
        {"name": "green_fp32", "kind": "green", "points": 4096, "prec": "fp32", "lam": 520.0, "theta": 0.35, "phi": 0.2,
         "a": 180.0, "b": 150.0, "z": 60.0},
        # the plain FP64 method on its smallest cell (a slab checked against the transfer matrix)
        {"name": "slab_fp64", "kind": "solve", "cell": "slab", "n": 6, "m": 2, "prec": "fp64", "lam": 500.0, "theta": 0.0,
         "phi": 0.0, "tol": 1e-8},
        # a coarse cell at conical incidence: latency of a whole solve
        {"name": "coarse_conical_fp32", "kind": "solve", "cell": "layered", "target": 774, "a": 200.0, "buffer": 40.0,
         "active": 100.0, "spheres": 1, "r": 20.0, "prec": "fp32", "lam": 560.0, "theta": 0.7, "phi": 0.2, "tol": 1e-6},
        # the enhancement study: a new cube cell per period, its first solve, with the absorption profile
        {"name": "cube_remesh_fp32", "kind": "remesh", "cell": "cube", "a": 80.0, "w": 40.0, "h": 10.0, "prec": "fp32",
         "lam": 560.0, "theta": 0.0, "phi": 0.0, "tol": 1e-6},
        # one point of the wavelength x angle sweep
        {"name": "sweep_point_fp32", "kind": "solve", "cell": "plasmonic", "h": 60.0, "hf": 14.5, "hz": 40.0, "prec": "fp32",
         "lam": 620.0, "theta": 0.5235987755982988, "phi": 0.0, "tol": 1e-6},
        # the sweep itself: angles 0..80 degrees in concurrent slots, 16-bit products
        {"name": "sweep_batch_fp16", "kind": "batch", "cell": "plasmonic", "h": 60.0, "hf": 14.5, "hz": 40.0, "prec": "fp16",
         "lam": 600.0, "points": 9, "slots": 3, "tol": 1e-6},
        # the headline solve
        {"name": "plasmonic_fp32", "kind": "solve", "cell": "plasmonic", "h": 30.0, "hf": 10.0, "hz": 25.0, "prec": "fp32",
         "lam": 500.0, "theta": 0.0, "phi": 0.0, "tol": 1e-6},
        # the same cell at conical incidence with BF16 products
        {"name": "plasmonic_conical_bf16", "kind": "solve", "cell": "plasmonic", "h": 30.0, "hf": 10.0, "hz": 25.0,
         "prec": "bf16", "lam": 500.0, "theta": 0.3, "phi": 0.5, "tol": 1e-6},
        # its refined mesh
        {"name": "plasmonic_fine_fp32", "kind": "solve", "cell": "plasmonic", "h": 28.0, "hf": 9.5, "hz": 25.0, "prec": "fp32",
         "lam": 500.0, "theta": 0.0, "phi": 0.0, "tol": 1e-6},
        # a burst of requests of different cells at a server
        {"name": "serve_fp32", "kind": "serve", "small": 2000, "large": 16000, "requests": 4, "slots": 3, "prec": "fp32",
         "tol": 1e-6},
        # the 2 x 2 sphere array over a metal grating, the largest cell that is solved in about a second
        {"name": "array_fp16", "kind": "solve", "cell": "array", "h": 40.0, "hf": 16.0, "hz": 27.0, "prec": "fp16",
         "lam": 600.0, "theta": 0.0, "phi": 0.0, "tol": 1e-6},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["green", "solve", "solve", "solve", "solve", "remesh", "batch", "serve"])
    prec = rng.choice(["fp32", "fp32", "fp32", "fp16", "bf16"])
    theta = rng.choice([0.0, rng.uniform(0.05, 1.3)])
    phi = rng.choice([0.0, rng.uniform(0.1, 1.4)])
    lam = rng.uniform(450.0, 780.0)
    if kind == "green":
        return {"kind": kind, "points": int(_log(rng, 1000, 300000)) | 1, "prec": rng.choice(["fp32", "fp32", "fp64"]),
                "lam": lam, "theta": theta, "phi": phi, "a": rng.uniform(120.0, 260.0), "b": rng.uniform(120.0, 260.0),
                "z": rng.uniform(30.0, 150.0)}
    if kind == "serve":
        return {"kind": kind, "small": int(_log(rng, 800, 4000)), "large": int(_log(rng, 4000, 14000)),
                "requests": rng.randint(2, 5), "slots": rng.randint(1, 4), "prec": prec, "tol": 1e-6}
    cell = {"cell": "layered", "target": int(_log(rng, 500, 26000 if kind == "solve" else 7000)),
            "a": rng.uniform(120.0, 260.0), "buffer": rng.uniform(30.0, 80.0), "active": rng.uniform(60.0, 130.0),
            "spheres": rng.choice([0, 1, 1]), "r": rng.uniform(14.0, 22.0)}
    if kind == "batch":
        return {"kind": kind, **cell, "prec": prec, "lam": lam, "points": rng.randint(3, 9), "slots": rng.randint(2, 4),
                "tol": 1e-6}
    if kind == "solve" and rng.random() < 0.12:   # the plain FP64 method, on slabs its Ewald series can afford
        return {"kind": kind, "cell": "slab", "n": rng.randint(3, 8), "m": rng.randint(1, 3), "prec": "fp64", "lam": lam,
                "theta": theta, "phi": phi, "tol": 1e-8}
    return {"kind": kind, **cell, "prec": prec, "lam": lam, "theta": theta, "phi": phi, "tol": 1e-6}


def _layered(target, a, buffer, active, spheres, r, seed):
    """A buffer and an active layer, a sphere in the middle of the active one, about `target` unknowns (2.05 per
    tetrahedron, six tetrahedra per grid cell)."""
    def cell(h):
        balls = [(0.5 * a, 0.5 * a, buffer + 0.5 * active, r, "ag")] if spheres else []
        return cellgen.layered_cell(a, a, [(buffer, "buffer"), (active, "active")], spheres=balls, h_coarse=h,
                                    h_fine=min(h, r / 1.2) if spheres else None, h_z=h, jitter=0.1, seed=seed,
                                    lateral_fine=target >= 2000)
    lo, hi = 2.0, 200.0
    for _ in range(12):
        mid = math.sqrt(lo * hi)
        lo, hi = (mid, hi) if 2.05 * cell(mid).n_tets > target else (lo, mid)
    return cell(hi)


def _cell(case, seed):
    if case["cell"] == "slab":
        return cellgen.slab_cell(case["n"], case["n"], case["m"], 200.0, 200.0, 40.0, (4.0, 0.5), jitter=0.1, seed=seed)
    if case["cell"] == "plasmonic":
        return cellgen.config_plasmonic(seed=seed, h_coarse=case["h"], h_fine=case["hf"], h_z=case["hz"])
    if case["cell"] == "cube":
        return cellgen.cube_cell(case["a"], 20.0, 60.0, case["w"], case["h"])
    if case["cell"] == "array":
        return cellgen.config_large(case["h"], case["hf"], case["hz"], seed=seed)
    return _layered(case["target"], case["a"], case["buffer"], case["active"], case["spheres"], case["r"], seed)


# What a program keeps of an answer.  The mixed paths hold the matrix and the Krylov vectors in single precision and
# stop at a residual of 1e-6, so their currents and fractions are stored in single precision; the FP64 path's in double.
def _currents(x, case):
    if isinstance(x, np.ndarray):
        return x if case["prec"] == "fp64" else x.astype(np.complex64)
    x = torch.view_as_complex(x)
    return x if case["prec"] == "fp64" else x.to(torch.complex64)


def _values(v, case):
    return np.asarray(v, dtype=np.float64 if case["prec"] == "fp64" else np.float32)


def _fractions(r, case):
    return {k: _values(r[k], case) for k in ("A", "R", "T")}


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    near = 1.0 + 0.004 * rng.uniform(-1.0, 1.0)   # the wavelength of this seed, within 0.4% of the case's
    if case["kind"] == "green":
        n = case["points"]
        d = rng.uniform(-0.999, 0.999, (n, 3)) * np.array([case["a"], case["b"], case["z"]])
        return {"case": case, "lib": vie.load(), "lam": case["lam"] * near, "d": torch.from_numpy(d).cuda(),
                "out": torch.empty((n, 2), dtype=torch.float64, device="cuda")}
    if case["kind"] == "serve":
        jobs = []
        for i in range(case["requests"]):
            f = i / max(1, case["requests"] - 1)
            cell = _layered(int(case["small"] * (case["large"] / case["small"]) ** f), 160.0 + 60.0 * f, 40.0 + 10.0 * i, 80.0,
                            i % 2, 20.0, seed + i)
            lam = (480.0 + 280.0 * f) * near
            jobs.append((cell, lam, 0.25 * i, 0.0, cell.eps(lam)))
        server = vie.Server(n_slots=case["slots"], precision=PREC[case["prec"]], tol=case["tol"])
        return {"case": case, "server": server, "jobs": jobs}
    cell = _cell(case, seed)
    solver = vie.Solver(precision=PREC[case["prec"]], tol=case["tol"])
    state = {"case": case, "solver": solver, "cell": cell, "lam": case["lam"] * near}
    n = solver.set_mesh(cell)
    if case["kind"] == "batch":
        k = case["points"]
        state["lams"] = [(case["lam"] + 5.0 * i) * near for i in range(k)]
        state["thetas"] = [math.radians(80.0 * i / max(1, k - 1)) for i in range(k)]
        state["eps"] = [cell.eps(l) for l in state["lams"]]
        return state
    state["eps"] = cell.eps(state["lam"])
    state["x"] = torch.empty((n, 2, 2), dtype=torch.float64, device="cuda")
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "green":
        rc = state["lib"].vie_green_noalloc(
            state["lam"], case["theta"], case["phi"], case["a"], case["b"], case["z"],
            ctypes.c_void_p(state["d"].data_ptr()), ctypes.c_void_p(state["out"].data_ptr()), case["points"],
            PREC[case["prec"]], ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc != 0:
            raise vie.VIEError(rc, "vie_green_noalloc")
        return {"g": torch.view_as_complex(state["out"])}
    if case["kind"] == "serve":
        tickets = [state["server"].submit(*job)[0] for job in state["jobs"]]
        done = [state["server"].poll(t) for t in tickets]
        return [_fractions(r, case) for r in done]
    solver = state["solver"]
    if case["kind"] == "batch":
        k = case["points"]
        out, _ = solver.solve_batch(state["lams"], state["thetas"], [0.0] * k, state["eps"], max_slots=case["slots"],
                                    coeffs=True)
        return [dict(_fractions(r, case), x=_currents(r["x"], case)) for r in out]
    if case["kind"] == "remesh":
        solver.set_mesh(state["cell"])
        r = solver.solve(state["lam"], case["theta"], case["phi"], state["eps"], coeffs=True, density=True)
        return dict(_fractions(r, case), x=_currents(r["x"], case), density=_values(r["density"], case))
    r = solver.solve_device(state["lam"], case["theta"], case["phi"], state["eps"], state["x"].data_ptr())
    nd = state["cell"].n_domains
    return {"A": _values([r.absorbed[0][:nd], r.absorbed[1][:nd]], case), "R": _values(r.reflectance[:], case),
            "T": _values(r.transmittance[:], case), "x": _currents(state["x"], case)}


def _solve_work(tets, size):
    """Filling the dense complex matrix (about 50 operations for each of the 16 tet-pair points, each unordered pair
    once) and one product with it for both polarisations; its entries are written and read once, and the currents
    (two complex doubles per unknown) come out."""
    n = 2.05 * tets
    return {"bytes": 2.0 * 2.0 * size * n * n + 32.0 * n, "flops": 50.0 * 8.0 * tets * tets + 16.0 * n * n}


def work(case):
    if case["kind"] == "green":
        # three coordinates in, one complex value out; about 50 terms of the two series, ten operations each
        return {"bytes": case["points"] * 40.0, "flops": case["points"] * 500.0}
    size = 8 if case["prec"] == "fp64" else 4
    if case["kind"] == "serve":
        k = case["requests"]
        each = [_solve_work(case["small"] * (case["large"] / case["small"]) ** (i / max(1, k - 1)) / 2.05, size)
                for i in range(k)]
        return {q: sum(w[q] for w in each) for q in ("bytes", "flops")}
    w = _solve_work(_cell(case, 0).n_tets, size)
    k = case["points"] if case["kind"] == "batch" else 1
    return {q: k * w[q] for q in w}


def _erfc(z):
    """erfc of complex z (numpy), Re z >= 0 by Weideman's rational expansion of w(iz) (SIAM J. Numer. Anal. 31, 1994)
    with 48 terms, Re z < 0 by erfc(-z) = 2 - erfc(z)."""
    n = 48
    big = math.sqrt(n / math.sqrt(2.0))
    t = big * np.tan(np.arange(-2 * n + 1, 2 * n) * math.pi / (4 * n))
    f = np.concatenate([[0.0], np.exp(-t * t) * (big * big + t * t)])
    a = np.real(np.fft.fft(np.fft.fftshift(f)))[1:n + 1] / (4 * n)
    u = np.where(z.real < 0, -z, z)
    q = (big - u) / (big + u)
    p = np.polyval(a[::-1], q)
    w = np.exp(-u * u) * (2.0 * p / (big + u) ** 2 + 1.0 / math.sqrt(math.pi) / (big + u))
    return np.where(z.real < 0, 2.0 - w, w)


def exact(case, seed):
    """The Green's functions by Ewald's two series in 64 bits.  The solves have no value that plain numpy reaches
    in 20 seconds: their matrix alone needs a second solver."""
    if case["kind"] != "green":
        return None
    s = prepare(case, seed)
    d = s["d"].cpu().numpy()
    x, y, z = d[:, 0], d[:, 1], np.abs(d[:, 2])
    a, b, k = case["a"], case["b"], 2.0 * math.pi / s["lam"]
    kx, ky = (k * math.sin(case["theta"]) * f(case["phi"]) for f in (math.cos, math.sin))
    e = math.sqrt(math.pi / (a * b))
    g = np.zeros(len(d), dtype=np.complex128)
    reach = 6.3
    for p in range(-12, 13):
        for q in range(-12, 13):
            tx, ty = kx + 2.0 * math.pi * p / a, ky + 2.0 * math.pi * q / b
            if math.hypot(tx, ty) > 2.0 * e * reach + k:
                continue
            gam = np.sqrt(complex(tx * tx + ty * ty - k * k))   # + j |gamma| for propagating orders
            t = np.exp(gam * z) * _erfc(gam / (2 * e) + z * e) + np.exp(-gam * z) * _erfc(gam / (2 * e) - z * e)
            g += np.exp(-1j * (tx * x + ty * y)) * t / (4.0 * a * b * gam)
    for m in range(-6, 7):
        for n in range(-6, 7):
            r = np.sqrt((x + m * a) ** 2 + (y + n * b) ** 2 + z * z)
            near = r * e < reach
            r = np.where(near, r, 1.0)
            c = np.exp(1j * k * r) * _erfc(r * e + 0.5j * k / e)
            g += np.where(near, np.exp(1j * (kx * m * a + ky * n * b)) * c.real / (4.0 * math.pi * r), 0.0)
    return {"g": g}
