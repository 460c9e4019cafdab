"""The same scatterers in other units of length.

Scaling all lengths by s and the wavenumbers by 1 / s leaves u as it is and
divides q by s, so every unit is checked against the dense oracle in the first
one.  The nodes are rounded anew in each unit, and the compression at tol 1e-12
is allowed 30 times tol as in the parity tests.  90 and 66 nodes: stages of 32
terms that hold both unknowns.
"""
import copy

import numpy as np
import pytest

from oracle import dense
from paper_2603_09381_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
ANGS = [0.3, 2.1, 4.0, 5.5]


@pytest.fixture(scope="module")
def pm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_09381_gb300 import pmchwt
    return pmchwt


def _scaled(prob, s):
    p = copy.deepcopy(prob)
    p["k_out"] /= s
    p["spacing"] *= s
    for c in p["inclusions"]:
        c["cx"], c["cy"], c["k_in"] = c["cx"] * s, c["cy"] * s, c["k_in"] / s
        c["prm"][0] *= s
        if c["shape"] == wl.SHAPE_ELLIPSE:
            c["prm"][1] *= s
    return p


def _unscaled(x, prob, s):
    x, o = x.copy(), 0
    for c in prob["inclusions"]:
        x[o:o + c["n"]] *= s
        o += 2 * c["n"]
    return x


def _problem(shape):
    prob = wl.star_grid(*{"one": (1, 1), "grid": (3, 2), "free": (2, 2)}[shape], n=66 if shape == "one" else 90, seed=3,
                        k_out=3.0)
    if shape == "free":   # an arbitrary arrangement with an ellipse
        prob["spacing"] = 0.0
        prob["inclusions"][2] = wl._inclusion(wl.SHAPE_ELLIPSE, 0.1, 1.2, 0.4, [0.42, 0.25], 72, 5.0)
    return prob


@pytest.mark.parametrize("e", [-9, -6, -3, -1.5, 0.8, 2, 5, 9])
@pytest.mark.parametrize("shape", ["one", "grid", "free"])
def test_solution_does_not_depend_on_the_unit(pm, shape, e):
    prob = _problem(shape)
    s = 10.0 ** e
    g = pm.Geometry(_scaled(prob, s))
    f = pm.Factor(g, 1e-12)
    F = g.plane_wave(ANGS)
    ref = dense.solve(prob, ANGS)
    for _ in range(2):   # eagerly, then from its graph
        x = _unscaled(f.solve(F), prob, s)
        assert np.linalg.norm(x - ref) < 3e-11 * np.linalg.norm(ref)


@pytest.mark.parametrize("s", [2.0 ** -20, 2.0 ** 20])
def test_a_power_of_two_changes_no_bit(pm, s):
    """... of u and of q times s; in a batch of several units, and on aliased device buffers too."""
    import torch
    prob = _problem("grid")
    g0, g1 = pm.Geometry(prob), pm.Geometry(_scaled(prob, s))
    x0 = pm.Factor(g0, 1e-10).solve(g0.plane_wave(ANGS))
    fs = pm.factor_batch([g1, g0], 1e-10, workers=1)
    F1 = g1.plane_wave(ANGS)
    x1 = pm.solve_batch(fs, [F1, g0.plane_wave(ANGS)], workers=1)
    # the mean radius is in [1/4, 1/2) in the first unit: both factor the same geometry
    assert np.array_equal(_unscaled(x1[0], prob, s), x0)
    f1 = pm.Factor(g1, 1e-10)
    y = f1.solve(F1)
    assert np.array_equal(y, x1[0]) and np.array_equal(x1[1], x0)
    d = torch.from_numpy(np.ascontiguousarray(F1.T)).cuda()
    f1.solve_device(d.data_ptr(), len(ANGS), d.data_ptr())
    torch.cuda.synchronize()
    assert np.array_equal(d.cpu().numpy().T, y)


def test_fields_nodes_and_blocks_keep_the_callers_unit(pm):
    prob = _problem("grid")
    s = 2.0 ** -20
    g0, g1 = pm.Geometry(prob), pm.Geometry(_scaled(prob, s))
    x0 = pm.Factor(g0, 1e-12).solve(g0.plane_wave(ANGS))
    x1 = pm.Factor(g1, 1e-12).solve(g1.plane_wave(ANGS))
    pts = np.array([[0.5, 3.0], [4.0, -2.0]])
    us0, us1 = g0.scattered_field(x0, pts), g1.scattered_field(x1, s * pts)
    assert np.linalg.norm(us1 - us0) < 1e-10 * np.linalg.norm(us0)
    assert np.array_equal(g1.nodes()[0], s * g0.nodes()[0])
    A0, A1 = g0.self_block(0, 90), g1.self_block(0, 90)
    assert np.array_equal(A1[:90, :90], s * A0[:90, :90])


@pytest.mark.parametrize("form", ["all", "bm"])
def test_other_formulations_in_other_units(pm, form):
    """Against the same formulation in the first unit (its discretisation is another one)."""
    prob = wl.star_grid(2, 1, n=66, seed=3, k_out=3.0)
    kw = {"formulation": {"all": pm.PM_FORM_ALL, "bm": pm.PM_FORM_BM}[form]}
    g0 = pm.Geometry(prob)
    ref = pm.Factor(g0, 1e-12, **kw).solve(g0.plane_wave(ANGS))
    for e in (-9, -3, 3, 9):
        s = 10.0 ** e
        g = pm.Geometry(_scaled(prob, s))
        x = _unscaled(pm.Factor(g, 1e-12, **kw).solve(g.plane_wave(ANGS)), prob, s)
        assert np.linalg.norm(x - ref) < 6e-11 * np.linalg.norm(ref)
