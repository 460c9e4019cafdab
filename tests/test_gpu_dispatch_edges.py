"""The solver at the edges of its dispatch rules: right-hand sides around the
groups of the field kernels and of the residual product, small ID matrices in
one launch or step by step, LU panels in shared memory or in place.
"""
import numpy as np
import pytest

from oracle import dense, field
from paper_2603_09381_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_09381_gb300 import pmchwt
    return pmchwt


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("nrhs", [1, 2, 3, 7, 8, 9, 15, 17])
def test_fields_in_groups_of_right_hand_sides(pm, nrhs):
    """Groups of 8, 4, 2 and 1: each column against the oracle's formulas on
    the same boundary values, and each column's bits whatever its group."""
    prob = wl.star_grid(3, 1, n=34, seed=4, k_out=4.0)
    g = pm.Geometry(prob)
    rng = np.random.default_rng(nrhs)
    phi = rng.standard_normal((g.N, nrhs)) + 1j * rng.standard_normal((g.N, nrhs))
    th = np.linspace(0, 6.2, 13)
    pts = np.stack([rng.uniform(-3, 6, 11), rng.uniform(1.0, 30.0, 11)], -1)   # both sides of k r = 8
    ff, us = g.far_field(phi, th), g.scattered_field(phi, pts)
    for c in range(nrhs):
        # sums of about 100 terms, each to a few 1e-15
        assert _rel(ff[:, c], field.far_field(prob, phi[:, c], th)) < 1e-13
        assert _rel(us[:, c], field.scattered_field(prob, phi[:, c], pts)) < 1e-12
        assert np.array_equal(ff[:, c], g.far_field(phi[:, c:c + 1], th)[:, 0])
        assert np.array_equal(us[:, c], g.scattered_field(phi[:, c:c + 1], pts)[:, 0])


@pytest.mark.parametrize("nx,ny,n,nrhs", [(2, 1, 32, 1), (2, 1, 34, 8), (3, 1, 66, 9), (2, 2, 70, 3), (3, 3, 62, 17)])
def test_mixed_residual_at_ragged_sizes(pm, nx, ny, n, nrhs):
    """The residual the refinement stops on is the true one (the oracle's
    matrix) at sizes that are no multiples of the product's tiles and with
    every size of its last group of right-hand sides."""
    prob = wl.star_grid(nx, ny, n=n, seed=2, k_out=4.0)
    angs = list(np.linspace(0.1, 6.0, nrhs))
    g = pm.Geometry(prob)
    F = g.plane_wave(angs)
    f = pm.Factor(g, 1e-10, precision=pm.PM_MIXED, refine_tol=1e-11)
    phi = f.solve(F)
    A = dense.assemble(prob)
    res = max(np.linalg.norm(F[:, r] - A @ phi[:, r]) / np.linalg.norm(F[:, r]) for r in range(nrhs))
    # entries agree to 1e-12 of their block's size
    assert f.last_info["residual"] <= 1e-11
    assert abs(res - f.last_info["residual"]) <= 5e-12


@pytest.mark.parametrize("mixed", [False, True])
def test_small_id_matrices_alone_and_in_a_large_group(pm, mixed):
    """Alone, a problem's ID matrices run all their steps in one launch; in a
    group of 48 they go step by step.  The same bits in complex128."""
    probs = [wl.circle_grid(2, 2, n=64, k_out=2.0 + 0.02 * i) for i in range(48)]
    gs = [pm.Geometry(p) for p in probs]
    kw = {"precision": pm.PM_MIXED, "refine_tol": 1e-11} if mixed else {}
    fs = pm.factor_batch(gs, 1e-10, workers=1, **kw)
    Fs = [g.plane_wave([0.4]) for g in gs]
    out = pm.solve_batch(fs, Fs, workers=1)
    for i in (0, 17, 47):
        x = pm.Factor(gs[i], 1e-10, **kw).solve(Fs[i])
        if mixed:   # both within the refined residual times the condition number (below 1e3 here)
            assert _rel(out[i], x) < 1e-8
        else:
            assert np.array_equal(out[i], x)
        assert _rel(x, dense.solve(probs[i], [0.4])) < 1e-8


@pytest.mark.parametrize("n", [520, 1740])
def test_tall_lu_panels(pm, n):
    """2 n rows: a panel in the shared memory of its cluster, and one that no longer fits."""
    prob = wl.star_grid(1, 1, n=n, seed=3, k_out=3.0)
    angs = [0.1, 2.5]
    g = pm.Geometry(prob)
    F = g.plane_wave(angs)
    x = pm.Factor(g, 1e-12).solve(F)
    A = dense.assemble(prob)
    # backward error: 2 n 2^-52 with a growth of ten, and entries that agree to 1e-12 of their block's size
    assert np.linalg.norm(A @ x - F) < 1e-11 * np.linalg.norm(A) * np.linalg.norm(x)


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4])
def test_solutions_for_few_waves(pm, nrhs, mixed):
    """One to three columns have a product kernel of their own, four do not;
    98 nodes a star leave rows past its 32-row blocks."""
    prob = wl.star_grid(2, 2, n=98, seed=6, k_out=4.0)
    angs = list(np.linspace(0.2, 5.0, nrhs))
    g = pm.Geometry(prob)
    kw = {"precision": pm.PM_MIXED, "refine_tol": 1e-11} if mixed else {}
    f = pm.Factor(g, 1e-12, **kw)
    F, ref = g.plane_wave(angs), dense.solve(prob, angs)
    assert _rel(f.solve(F), ref) < (1e-8 if mixed else 3e-11)
    assert _rel(f.solve(F), ref) < (1e-8 if mixed else 3e-11)   # replayed from its graph
