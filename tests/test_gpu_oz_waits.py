"""A bounded wait of the FP64-accurate tensor-core products that runs out.

Each CTA first waits, with a bound of about a millisecond, on a barrier that
nothing arrives at; it then cuts, issues and stores nothing, drains, frees its
tensor memory and flags the error.  The call returns PM_ERR_TIMEOUT, and the
next one works.
"""
import numpy as np
import pytest

from oracle import dense
from paper_2603_09381_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pm():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_09381_gb300 import pmchwt
    return pmchwt


def _still_solves(pm, prob, angs):
    g = pm.Geometry(prob)
    x = pm.Factor(g, 1e-10).solve(g.plane_wave(angs))
    ref = dense.solve(prob, angs)
    return np.linalg.norm(x - ref) < 1e-8 * np.linalg.norm(ref)


# 70 nodes: QR panels with trailing columns; one inclusion: LU updates of several stages
@pytest.mark.parametrize("nx,n,mixed", [(2, 96, False), (1, 70, False), (2, 64, True)])
def test_a_wait_of_the_factorization_that_runs_out(pm, nx, n, mixed):
    prob = wl.star_grid(nx, 1, n=n, seed=1, k_out=3.0)
    g = pm.Geometry(prob)
    with pytest.raises(pm.PmError) as e:
        pm.Factor(g, 1e-10, precision=pm.PM_MIXED if mixed else pm.PM_FP64, debug_flags=pm.PM_DEBUG_OZ_NO_ARRIVE)
    assert e.value.status == 6
    assert _still_solves(pm, prob, [0.5])


# FP64: Schur products (4 columns) and blocked triangles (65); mixed: the residual product
@pytest.mark.parametrize("nrhs,mixed", [(4, False), (65, False), (2, True)])
def test_a_wait_of_the_solve_that_runs_out(pm, nrhs, mixed):
    prob = wl.star_grid(2, 1, n=64, seed=1, k_out=3.0)
    angs = list(np.linspace(0.2, 6.0, nrhs))
    g = pm.Geometry(prob)
    f = pm.Factor(g, 1e-10, precision=pm.PM_MIXED if mixed else pm.PM_FP64, debug_flags=pm.PM_DEBUG_OZ_SOLVE_NO_ARRIVE)
    for _ in range(2):   # the factor stays usable: the second call reports the same
        with pytest.raises(pm.PmError) as e:
            f.solve(g.plane_wave(angs))
        assert e.value.status == 6
    assert _still_solves(pm, prob, angs)
