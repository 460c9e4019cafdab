"""The solver's work as its users have it done, case by case, for timing.

Each case is one call sequence through the Python entry points (pmchwt.py):
factor a configuration and solve for a few incident waves, solve again with a
kept factorization, factor and solve a batch, evaluate fields.  Geometry
handles, right-hand sides on the device and the trained predictor are what a
program has in hand before; the factorization is made anew in every pass.
"""
import math

import numpy as np
import torch

from paper_2603_09381_gb300 import pmchwt as pm
from paper_2603_09381_gb300 import rank_predictor

CIRCLE, ELLIPSE, STAR, FOURIER = 0, 1, 2, 3
FORMS = {"omit": pm.PM_FORM_OMIT, "all": pm.PM_FORM_ALL, "bm": pm.PM_FORM_BM}


# ---------------------------------------------------------------- the cases

def _direct(name, shape, nx, ny, n, tol=1e-10, precision="fp64", nrhs=8, k=2 * math.pi * 20 / 16, ratio=2.0,
            lossy=False, form="omit", proxy=0, predictor=False, whole=False):
    return {"name": name, "op": "direct", "shape": shape, "nx": nx, "ny": ny, "n": n, "tol": tol,
            "precision": precision, "nrhs": nrhs, "k": k, "ratio": ratio, "lossy": lossy, "form": form,
            "proxy": proxy, "predictor": predictor, "whole": whole}


def listed():
    return [
        # the 2 x 2 disks of the closed-form check, from descriptors to a host
        # solution in one go: the smallest problem, all latency
        _direct("disks2_fp64", "circles", 2, 2, 64, tol=1e-12, nrhs=1, k=2 * math.pi, proxy=64, whole=True),
        # the same disks with an absorbing interior in mixed precision
        _direct("disks2_lossy_mixed", "circles", 2, 2, 64, tol=1e-12, precision="mixed", nrhs=1, k=2 * math.pi,
                lossy=True, proxy=64),
        # a 4 x 4 block of the 16 x 16 stars, FP64, eight waves
        _direct("stars4_fp64", "stars", 4, 4, 128),
        # ragged grid of random smooth shapes with a contrast of its own each
        _direct("fourier7x5_fp64", "fourier", 7, 5, 96, k=5.0, ratio=0.0, nrhs=3),
        # ellipses anywhere (not on a grid), one wave
        _direct("scattered20_fp64", "anywhere", 20, 1, 96, k=2 * math.pi, nrhs=1),
        # Burton-Miller at omega = 5, eps- = 5 (the formulation comparison)
        _direct("stars3x4_bm_fp64", "stars", 3, 4, 128, k=5.0, ratio=math.sqrt(5.0), form="bm", nrhs=2),
        # FP64 at 16,384 unknowns: the plain solver where it is compute-bound
        _direct("stars8_fp64", "stars", 8, 8, 128),
        # mixed precision with the trained predictor: 8 x 8 and the full 16 x 16 stars (65,536 unknowns)
        _direct("stars8_mixed", "stars", 8, 8, 128, precision="mixed", predictor=True),
        _direct("stars16_mixed", "stars", 16, 16, 128, precision="mixed", predictor=True),
        # independent ellipse problems of uneven sizes in shared launches, host buffers
        {"name": "ellipses_batch_mixed", "op": "batch", "count": 12, "m_lo": 4, "m_hi": 32, "tol": 1e-10,
         "precision": "mixed", "nrhs": 2, "workers": 4, "layout": 1},
        # a kept FP64 factorization solved for a new set of incident waves
        {"name": "resolve_fp64", "op": "resolve", "shape": "stars", "nx": 5, "ny": 5, "n": 128, "tol": 1e-10,
         "precision": "fp64", "nrhs": 16, "k": 2 * math.pi * 20 / 16, "ratio": 2.0},
        # near and far field of eight solutions: an observation window and all directions
        {"name": "fields_stars8", "op": "fields", "shape": "stars", "nx": 8, "ny": 8, "n": 128, "nrhs": 8,
         "k": 2 * math.pi * 20 / 16, "ratio": 2.0, "points": 4096, "directions": 720},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["fp64", "fp64", "fp64", "mixed", "mixed", "batch", "resolve", "fields"])
    if op == "batch":
        return {"op": "batch", "count": rng.randint(3, 12), "m_lo": 2, "m_hi": _log_int(rng, 4, 32), "tol": 1e-10,
                "precision": rng.choice(["mixed", "mixed", "fp64"]), "nrhs": rng.randint(1, 4),
                "workers": rng.choice([2, 4]), "layout": rng.randint(2, 999)}
    shape = rng.choice(["stars", "stars", "fourier", "circles", "anywhere"])
    n = 2 * _log_int(rng, 16, 72)
    most = {"fp64": 48, "mixed": 160, "resolve": 25, "fields": 64}[op]   # inclusions
    m = _log_int(rng, 2, most)
    if shape == "anywhere":
        nx, ny = min(m, 40), 1
    else:
        nx = max(1, int(round(math.sqrt(m) * rng.uniform(0.75, 1.3))))
        ny = max(1, m // nx)
        if nx * ny == 1:
            nx = 2
    k = rng.uniform(2.0, 8.0)
    n = max(n, 32, 2 * int(math.ceil(5 * k)))   # enough nodes for the interior wavelength
    geo = {"shape": shape, "nx": nx, "ny": ny, "n": n, "k": k,
           "ratio": 0.0 if shape == "fourier" else rng.uniform(1.5, 2.2)}
    if op == "fields":
        return {"op": "fields", **geo, "nrhs": rng.randint(1, 8), "points": _log_int(rng, 100, 4096),
                "directions": _log_int(rng, 30, 720)}
    if op == "resolve":
        return {"op": "resolve", **geo, "tol": 1e-10, "precision": rng.choice(["fp64", "mixed"]),
                "nrhs": rng.choice([1, 2, 3, 5, 8, 16, 33])}
    form = "omit"
    if op == "fp64" and shape in ("stars", "circles") and rng.random() < 0.3:
        form = rng.choice(["all", "bm"])
    if form != "omit":   # four to six times the ID work: fewer inclusions
        geo["nx"], geo["ny"] = min(nx, 4), min(ny, 4)
    c = _direct("", **geo, tol=10 ** rng.uniform(-12, -10), precision=op, nrhs=rng.choice([1, 2, 3, 5, 8, 16]),
                form=form, predictor=op == "mixed" and rng.random() < 0.5, whole=rng.random() < 0.2)
    del c["name"]
    return c


# ------------------------------------------------------- problems and inputs

def _problem(case, rng):
    """Descriptor dictionary of a configuration (rotations, shapes and contrasts from rng)."""
    k, n, shape = case["k"], case["n"], case["shape"]
    centres = [(float(ix), float(iy)) for iy in range(case["ny"]) for ix in range(case["nx"])]
    spacing, sizes = 1.0, None
    if shape == "anywhere":
        m = case["nx"] * case["ny"]
        box, gap, centres, sizes = 1.15 * math.sqrt(m) + 0.5, 0.12, [], []
        while len(centres) < m:
            a, b = rng.uniform(0.2, 0.4, size=2)
            for _ in range(200):
                c = rng.uniform(0.0, box, size=2)
                if all(math.hypot(c[0] - x, c[1] - y) >= max(a, b) + max(s) + gap
                       for (x, y), s in zip(centres, sizes)):
                    centres.append((float(c[0]), float(c[1])))
                    sizes.append((float(a), float(b)))
                    break
            else:
                box *= 1.1
        spacing = 0.0
    inc = []
    for j, (cx, cy) in enumerate(centres):
        rot, k_in = 0.0, case["ratio"] * k
        if shape == "circles":
            kind, prm = CIRCLE, [0.4]
        elif shape == "stars":
            kind, prm, rot = STAR, [0.4, 0.2, 5.0], rng.uniform(0.0, 2 * math.pi / 5)
        elif shape == "fourier":
            kind = FOURIER
            prm = [0.4, *rng.uniform(0.0, 0.04, size=5), *rng.uniform(0.0, 2 * math.pi, size=5)]
        else:
            a, b = sizes[j] if sizes else rng.uniform(0.2, 0.45, size=2)
            kind, prm, rot = ELLIPSE, [a, b], rng.uniform(0.0, math.pi)
        if not case["ratio"]:
            k_in = rng.uniform(1.5, 3.0) * k
        prm = [float(v) for v in prm]
        inc.append({"shape": kind, "cx": cx, "cy": cy, "rot": float(rot), "prm": prm + [0.0] * (16 - len(prm)),
                    "n": n, "k_in": complex(k_in) * (1 + 0.05j if case.get("lossy") else 1)})
    return {"k_out": float(k), "inclusions": inc, "grid_nx": case["nx"], "grid_ny": case["ny"], "spacing": spacing}


def _batch_problems(case, rng):
    out, sizes = [], np.random.default_rng(case["layout"])
    for _ in range(case["count"]):
        m = int(sizes.integers(case["m_lo"], case["m_hi"] + 1))
        cols = int(math.ceil(math.sqrt(m)))
        n = int(sizes.choice(np.arange(64, 129, 32)))
        k = 2 * math.pi * rng.uniform(0.5, 1.4)   # wavelengths per spacing
        c = {"shape": "ellipses", "nx": cols, "ny": int(math.ceil(m / cols)), "n": n, "k": k, "ratio": 0.0}
        p = _problem(c, rng)
        p["inclusions"] = p["inclusions"][:m]
        out.append(p)
    return out


def _nodes(inc):
    """Positions, unit normals, speed, (n . x'') / |x'| at the n equispaced parameters of one curve."""
    n, p = inc["n"], inc["prm"]
    t = 2 * math.pi * np.arange(n) / n
    c, s = np.cos(t), np.sin(t)
    if inc["shape"] == ELLIPSE:
        x, d, e = (np.stack(v) for v in ((p[0] * c, p[1] * s), (-p[0] * s, p[1] * c), (-p[0] * c, -p[1] * s)))
    else:
        if inc["shape"] == CIRCLE:
            terms = []
        elif inc["shape"] == STAR:
            terms = [(p[1], p[2], 0.0)]
        else:
            terms = [(p[m - 1], float(m), p[m + 4]) for m in range(2, 7)]
        r, r1, r2 = np.ones(n), np.zeros(n), np.zeros(n)
        for a, m, ph in terms:
            r, r1, r2 = (r + a * np.cos(m * t + ph), r1 - a * m * np.sin(m * t + ph),
                         r2 - a * m * m * np.cos(m * t + ph))
        z = p[0] * np.exp(1j * t)
        z0, z1, z2 = r * z, (r1 + 1j * r) * z, (r2 + 2j * r1 - r) * z
        x, d, e = (np.stack((v.real, v.imag)) for v in (z0, z1, z2))
    cr, sr = math.cos(inc["rot"]), math.sin(inc["rot"])
    q = np.array([[cr, -sr], [sr, cr]])
    x, d, e = q @ x + np.array([[inc["cx"]], [inc["cy"]]]), q @ d, q @ e
    speed = np.hypot(d[0], d[1])
    nrm = np.stack((d[1], -d[0])) / speed
    return x, nrm, speed, (nrm * e).sum(0) / speed


def _waves(prob, angles):
    """Right-hand sides [-u^I; -q^I] per inclusion for plane waves, one row per angle."""
    k, rows = prob["k_out"], []
    for a in angles:
        d = np.array([math.cos(a), math.sin(a)])
        parts = []
        for inc in prob["inclusions"]:
            x, nrm, _, _ = _nodes(inc)
            u = np.exp(1j * k * (d @ x))
            parts += [-u, -1j * k * (d @ nrm) * u]
        rows.append(np.concatenate(parts))
    return np.stack(rows)


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    if case["op"] == "batch":
        probs = _batch_problems(case, rng)
        return probs, [_waves(p, rng.uniform(0, 2 * math.pi, case["nrhs"])) for p in probs]
    prob = _problem(case, rng)
    return prob, _waves(prob, rng.uniform(0, 2 * math.pi, case["nrhs"]))


def _window(case, prob, seed):
    """Observation points above the configuration and far-field directions."""
    rng = np.random.default_rng([seed, 1])
    top = max(c["cy"] for c in prob["inclusions"]) + 0.9
    xs = [c["cx"] for c in prob["inclusions"]]
    pts = np.stack([rng.uniform(min(xs) - 1, max(xs) + 1, case["points"]),
                    rng.uniform(top, top + 4.0, case["points"])], 1)
    return pts, np.sort(rng.uniform(0, 2 * math.pi, case["directions"]))


# ------------------------------------------------------------ prepare and run

def _options(case, model):
    o = {"precision": pm.PM_MIXED if case["precision"] == "mixed" else pm.PM_FP64}
    if case["precision"] == "mixed":   # a residual that leaves the solution itself ten digits
        o["refine_tol"] = 1e-11
    if "form" in case:
        o.update(formulation=FORMS[case["form"]], proxy_points=case["proxy"])
    if model is not None:
        o["rank_model"] = model.data_ptr()
    return o


def prepare(case, seed):
    if case["op"] == "batch":
        probs, rhs = _inputs(case, seed)
        return {"case": case, "geoms": [pm.Geometry(p) for p in probs], "rhs": [r.T for r in rhs]}
    prob, rhs = _inputs(case, seed)
    s = {"case": case, "prob": prob}
    if case.get("predictor"):
        s["model"] = rank_predictor.to_device(rank_predictor.load_model())
    if case.get("whole"):   # the run starts from the descriptors and host arrays
        s["rhs"] = rhs.T
        return s
    s["geom"] = pm.Geometry(prob)
    if case["op"] == "fields":
        s["phi"] = _traces(prob, rhs).T
        s["points"], s["angles"] = _window(case, prob, seed)
        return s
    s["rhs"] = torch.from_numpy(rhs).cuda()      # nrhs x N: N x nrhs column-major
    if case["op"] == "resolve":
        s["factor"] = pm.Factor(s["geom"], case["tol"], **_options(case, None))
    return s


def run(s):
    case = s["case"]
    if case["op"] == "batch":
        fs = pm.factor_batch(s["geoms"], case["tol"], workers=case["workers"], **_options(case, None))
        return pm.solve_batch(fs, s["rhs"], workers=case["workers"])
    if case["op"] == "fields":
        return [s["geom"].scattered_field(s["phi"], s["points"]), s["geom"].far_field(s["phi"], s["angles"])]
    if case.get("whole"):
        f = pm.Factor(pm.Geometry(s["prob"]), case["tol"], **_options(case, s.get("model")))
        return f.solve(s["rhs"])
    f = s["factor"] if case["op"] == "resolve" else pm.Factor(s["geom"], case["tol"],
                                                              **_options(case, s.get("model")))
    rhs = s["rhs"]
    phi = torch.empty_like(rhs)
    f.solve_device(rhs.data_ptr(), rhs.shape[0], phi.data_ptr())
    return phi


def _traces(prob, waves):
    """Boundary values [q; u] for the field kernels, one row per wave: the incident wave's traces
    with half of u (with all of it the represented field vanishes outside)."""
    out, o = np.empty_like(waves), 0
    for inc in prob["inclusions"]:
        n = inc["n"]
        out[:, o:o + n], out[:, o + n:o + 2 * n] = -waves[:, o + n:o + 2 * n], -0.5 * waves[:, o:o + n]
        o += 2 * n
    return out


# --------------------------------------------------------------------- work

def _solver_work(prob, tol, nrhs, form="omit", factor=True):
    """Floating-point operations of the compressed solver on a configuration, by the usual
    counts: kernel entries and Householder IDs to a rank that grows with a box's perimeter, LU
    and Schur products per box, the top LU, the triangular solves."""
    m = len(prob["inclusions"])
    n = prob["inclusions"][0]["n"]
    flops, mats, lev, boxes, cand = 0.0, 0.0, 0, float(m), float(n)
    fam = 1.0 if form == "omit" else 2.0
    digits = -math.log10(tol) / 10
    while boxes > 1:
        side = 2.0 ** lev
        rank = min(cand, (28 + 60 * side) * digits * (1.0 if form == "omit" else 1.4))
        near = min(4.0, boxes - 1)
        rows = near * 2 * cand + 2 * fam * (2 * prob["k_out"] * 1.5 * 0.75 * side + 57 * digits)
        mb, kb = 2 * cand, 2 * rank
        ident = 16 * rows * cand * rank - 8 * (rows + cand) * rank ** 2 + 16 / 3 * rank ** 3
        flops += boxes * 4 * (100 * rows * cand * fam + max(ident, 0.0))
        flops += boxes * (8 / 3 * mb ** 3 + 8 * mb * mb * kb + 8 * mb * kb * kb + 32 / 3 * kb ** 3)
        mats += boxes * (mb * mb + 2 * mb * kb + kb * kb)
        cand, boxes, lev = min(4.0, boxes) * rank, math.ceil(boxes / 4), lev + 1
    top = 2 * cand
    flops += 8 / 3 * top ** 3
    mats += top * top
    solve = 8 * mats * nrhs
    return (flops if factor else 0.0) + solve, mats


def work(case):
    if case["op"] == "batch":
        c = {"shape": "ellipses", "n": 96, "k": 6.0, "ratio": 2.0}
        m = (case["m_lo"] + case["m_hi"]) / 2
        c["nx"] = c["ny"] = max(1, int(round(math.sqrt(m))))
        prob = _problem(c, np.random.default_rng(0))
        N = 2 * 96 * m
        return {"bytes": case["count"] * 32.0 * N * case["nrhs"],
                "flops": case["count"] * _solver_work(prob, case["tol"], case["nrhs"])[0]}
    prob = _problem(case, np.random.default_rng(0))
    N = sum(2 * c["n"] for c in prob["inclusions"])
    if case["op"] == "fields":
        # about 60 operations for a Hankel pair or a sincos, 16 a right-hand side
        per = 60.0 + 16.0 * case["nrhs"]
        return {"bytes": 16.0 * case["nrhs"] * (N + case["points"] + case["directions"]),
                "flops": per * N / 2 * (case["points"] + case["directions"])}
    kept = case["op"] == "resolve"
    flops, mats = _solver_work(prob, case["tol"], case["nrhs"], case.get("form", "omit"), factor=not kept)
    if case["precision"] == "mixed":   # the FP64 operator's entries, and its product once
        flops += (100.0 / 4 if not kept else 0.0) * N * N / 2 + 8.0 * N * N * case["nrhs"]
    return {"bytes": 32.0 * N * case["nrhs"] + (16.0 * mats if kept else 0.0), "flops": flops}


# ----------------------------------------------- what 64-bit arithmetic gives

def _hankel(z):
    """J0, J1, H0, H1: backward recurrence and Neumann's series for Y below 18, the asymptotic
    expansion from there on (real arguments only)."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    z = torch.as_tensor(z).to(dev)
    small = z if z.is_complex() else z.clamp(max=18.0)
    hi, lo = torch.zeros_like(small), torch.full_like(small, 1e-250)   # J_61, J_60 up to a factor
    norm, s0, s1 = torch.zeros_like(small), torch.zeros_like(small), torch.zeros_like(small)
    for m in range(60, 0, -1):      # lo is J_m here
        if m % 2 == 0:
            norm += 2 * lo
            s0 += (-1) ** (m // 2) / (m // 2) * lo
        elif m > 1:
            k = m // 2
            s1 += (-1) ** k * m / (k * (k + 1)) * lo
        hi, lo = lo, (2 * m) * lo / small - hi
    norm += lo
    j0, j1, s0, s1 = lo / norm, hi / norm, s0 / norm, s1 / norm
    lg = torch.log(small / 2) + np.euler_gamma
    y0 = (2 * lg * j0 - 4 * s0) / math.pi
    y1 = (-2 * j0 / small + 2 * (lg - 1) * j1 - 2 * s1) / math.pi
    h0, h1 = j0 + 1j * y0, j1 + 1j * y1
    if not z.is_complex():
        big = z.clamp(min=18.0)
        for nu in (0, 1):
            t = torch.ones_like(big) + 0j
            acc = t.clone()
            for m in range(1, 30):
                t = t * (1j * (4 * nu * nu - (2 * m - 1) ** 2) / (8.0 * m)) / big
                acc += t
            h = torch.sqrt(2 / (math.pi * big)) * torch.exp(1j * (big - math.pi / 4)) * ((-1j) ** nu * acc)
            if nu == 0:
                h0 = torch.where(z < 18, h0, h)
            else:
                h1 = torch.where(z < 18, h1, h)
        j0, j1 = h0.real, h1.real
    return j0, j1, h0, h1


def _self_operators(nd, k):
    """S, D, D*, N of one curve: Kress's log-split rule and Maue's identity."""
    x, nrm, speed, curv = nd
    n = len(speed)
    M, h = n // 2, 2 * math.pi / n
    i = np.arange(n)
    diff = i[:, None] - i[None, :]
    off = diff != 0
    s = h * i
    R = sum(np.cos(m * s) / m for m in range(1, M)) * (-2 * math.pi / M) - (math.pi / M ** 2) * np.cos(M * s)
    R = R[diff % n]
    lg = np.log(4 * np.sin(h * diff / 2) ** 2 + ~off)
    d = x[:, :, None] - x[:, None, :]
    r = np.where(off, np.hypot(d[0], d[1]), 1.0)
    j0, j1, h0, h1 = (v.cpu().numpy() for v in _hankel(k.real * r if k.imag == 0 else k * r))
    k = k.real if k.imag == 0 else k
    cos_y = (nrm[0][None] * d[0] + nrm[1][None] * d[1]) / r
    cos_x = (nrm[0][:, None] * d[0] + nrm[1][:, None] * d[1]) / r
    w = speed[None, :]
    di = np.arange(n)

    def split(full, log_part, diag_log, diag_smooth):
        log_part = np.where(off, log_part, 0.0)
        smooth = np.where(off, full - log_part * lg, 0.0).astype(np.complex128)
        log_part = log_part.astype(np.complex128)
        log_part[di, di], smooth[di, di] = diag_log, diag_smooth
        return R * log_part + h * smooth

    S = split(0.25j * h0 * w, -j0 * w / (4 * math.pi), -speed / (4 * math.pi),
              (0.25j - (np.euler_gamma + np.log(k * speed / 2)) / (2 * math.pi)) * speed)
    D = split(0.25j * k * h1 * cos_y * w, -k / (4 * math.pi) * j1 * cos_y * w, 0.0, curv / (4 * math.pi))
    Ds = split(-0.25j * k * h1 * cos_x * w, k / (4 * math.pi) * j1 * cos_x * w, 0.0, curv / (4 * math.pi))
    T = np.where(off, 0.5 * (-1.0) ** diff / np.tan(h * diff / 2 + ~off), 0.0)
    N = (T @ (S / w) @ T) / speed[:, None] + k * k * S * (nrm.T @ nrm)
    return S, D, Ds, N


def _far_operators(x, nrm, w, k):
    """S, D, D*, N between all nodes by the trapezoid rule (the diagonal means nothing)."""
    d = x[:, :, None] - x[:, None, :]
    r = torch.sqrt(d[0] ** 2 + d[1] ** 2)
    r.fill_diagonal_(1.0)
    _, _, h0, h1 = _hankel(k * r)
    cy = (nrm[0][None] * d[0] + nrm[1][None] * d[1]) / r
    cx = (nrm[0][:, None] * d[0] + nrm[1][:, None] * d[1]) / r
    del d
    g = 0.25j * k * w[None, :]
    return (g / k * h0, g * h1 * cy, -g * h1 * cx,
            g * (k * h0 * cx * cy + h1 / r * (nrm.T @ nrm - 2 * cx * cy)))


def _system(prob, form):
    k0, incs = prob["k_out"], prob["inclusions"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    nds = [_nodes(c) for c in incs]
    off = np.concatenate([[0], np.cumsum([2 * c["n"] for c in incs])])
    x, nrm = (torch.from_numpy(np.concatenate([nd[i] for nd in nds], 1)).to(dev) for i in (0, 1))
    w = torch.from_numpy(np.concatenate([2 * math.pi / len(nd[2]) * nd[2] for nd in nds])).to(dev)
    first = torch.from_numpy(np.concatenate([o + np.arange(c["n"]) for o, c in zip(off, incs)])).to(dev)
    second = torch.from_numpy(np.concatenate([o + c["n"] + np.arange(c["n"]) for o, c in zip(off, incs)])).to(dev)
    A = torch.empty((int(off[-1]),) * 2, dtype=torch.complex128, device=dev)
    al = 1j / k0
    S, D, Ds, N = _far_operators(x, nrm, w, k0)
    if form == "omit":
        blk = [[-S, D], [-Ds, N]]
    else:
        ki = incs[0]["k_in"].real
        ei = (ki / k0) ** 2
        s, d, ds, nn = _far_operators(x, nrm, w, ki)
        blk = ([[D + al * N, -(S + al * Ds)], [d, -ei * s]] if form == "bm" else
               [[-(S + ei * s), D + d], [-(Ds + ds), N + nn / ei]])
    for rows, line in zip((first, second), blk):
        for cols, b in zip((first, second), line):
            A[rows[:, None], cols[None, :]] = b
    del blk, S, D, Ds, N
    seen = {}
    for i, c in enumerate(incs):
        ki, ei = c["k_in"], (c["k_in"] / k0) ** 2
        key = repr((c["shape"], c["prm"], c["rot"], c["n"], ki))
        if key not in seen:
            S, D, Ds, N = _self_operators(nds[i], complex(k0))
            s, d, ds, nn = _self_operators(nds[i], ki)
            if form == "bm":
                e = 0.5 * np.eye(c["n"])
                b = np.block([[D - e + al * N, -S - al * (Ds + e)], [d + e, -ei * s]])
            else:
                b = np.block([[-(S + ei * s), D + d], [-(Ds + ds), N + nn / ei]])
            seen[key] = torch.from_numpy(b).to(dev)
        A[off[i]:off[i + 1], off[i]:off[i + 1]] = seen[key]
    return A, off


def _dense_solution(prob, rhs, form="omit"):
    """phi (N x nrhs) of the dense Nystrom system."""
    A, off = _system(prob, form)
    F = rhs.T.copy()
    if form == "bm":
        al = 1j / prob["k_out"]
        for o, c in zip(off, prob["inclusions"]):
            n = c["n"]
            F[o:o + n] += al * F[o + n:o + 2 * n]
            F[o + n:o + 2 * n] = 0
    lu = torch.linalg.lu_factor(A)
    b = torch.from_numpy(F).to(A.device)
    X = torch.linalg.lu_solve(*lu, b)
    X = (X + torch.linalg.lu_solve(*lu, b - A @ X)).cpu().numpy()
    if form == "bm":
        Y = X.copy()
        for o, c in zip(off, prob["inclusions"]):
            n = c["n"]
            Y[o:o + n], Y[o + n:o + 2 * n] = X[o + n:o + 2 * n], X[o:o + n]
        X = Y
    return X


def _fields(prob, phi, pts, angles):
    k = prob["k_out"]
    us = np.zeros((len(pts), phi.shape[0]), np.complex128)
    ff = np.zeros((len(angles), phi.shape[0]), np.complex128)
    xh, o = np.stack((np.cos(angles), np.sin(angles))), 0
    gamma = 0.25j * math.sqrt(2 / (math.pi * k)) * np.exp(-0.25j * math.pi)
    for c in prob["inclusions"]:
        n = c["n"]
        y, nrm, speed, _ = _nodes(c)
        w = 2 * math.pi / n * speed
        q, u = phi[:, o:o + n].T * w[:, None], phi[:, o + n:o + 2 * n].T * w[:, None]
        d = pts.T[:, :, None] - y[:, None, :]
        r = np.hypot(d[0], d[1])
        h0, h1 = (v.cpu().numpy() for v in _hankel(k * r)[2:])
        us += 0.25j * (k * h1 * (nrm[0][None] * d[0] + nrm[1][None] * d[1]) / r) @ u - 0.25j * h0 @ q
        pw = np.exp(-1j * k * (xh.T @ y))
        ff += gamma * ((pw * (-1j * k * (xh.T @ nrm))) @ u - pw @ q)
        o += 2 * n
    return [us, ff]


def exact(case, seed):
    if case["op"] == "batch":
        probs, rhs = _inputs(case, seed)
        sizes = [sum(2 * c["n"] for c in p["inclusions"]) for p in probs]
        if sum(v ** 2 for v in sizes) > 1.5e8:
            return None
        return [_dense_solution(p, r) for p, r in zip(probs, rhs)]
    prob, rhs = _inputs(case, seed)
    if case["op"] == "fields":
        return _fields(prob, _traces(prob, rhs), *_window(case, prob, seed))
    if rhs.shape[1] > 9000:
        return None
    X = _dense_solution(prob, rhs, case.get("form", "omit"))
    return X if case.get("whole") else torch.from_numpy(np.ascontiguousarray(X.T))
