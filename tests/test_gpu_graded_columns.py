"""The refinement's residual product with inclusions of very different sizes.

The columns of small inclusions hold large entries of the operator and meet
small entries of X.  The refinement has to reach a residual of 1e-11 as it
does with the operator applied in FP64, and the two solutions agree to both
residuals times the condition number (below 1e4 here).
"""
import numpy as np
import pytest

from paper_2603_09381_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("f,n,nrhs", [(0.03, 90, 4), (0.02, 90, 4), (0.03, 70, 9), (0.1, 64, 1)])
def test_refinement_reaches_its_tolerance_with_small_inclusions(f, n, nrhs):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_09381_gb300 import pmchwt as pm
    prob = wl.star_grid(3, 3, n=n, seed=3, k_out=3.0)
    for i, c in enumerate(prob["inclusions"]):
        if i % 2:
            c["prm"][0] *= f
    g = pm.Geometry(prob)
    F = g.plane_wave(list(np.linspace(0.3, 5.5, nrhs)))
    kw = {"precision": pm.PM_MIXED, "refine_tol": 1e-11, "max_refine": 14}
    fac = pm.Factor(g, 1e-10, **kw)
    x = fac.solve(F)
    assert fac.last_info["residual"] <= 1e-11
    y = pm.Factor(g, 1e-10, dense_operator=False, **kw).solve(F)
    assert np.linalg.norm(x - y) < 2e-7 * np.linalg.norm(y)
