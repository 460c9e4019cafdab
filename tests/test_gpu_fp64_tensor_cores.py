"""FP64 products on the tensor cores (integer digits, FP64 accuracy): LU, LU
solves and batched products at the edges of their 128 x 32 tiles and 32-deep
stages, and the QR-first reduction of complex128 ID inputs at the edges of
its 32-column panels.

A single inclusion is one dense LU of 2 n unknowns, so the solver and the
dense oracle factor the same matrix: both are backward stable, and the
difference is bounded by the condition number (below 1e4 at these sizes)
times n times 2^-52, 1e-10 with a wide margin.  Several inclusions add the
compression at tol 1e-12, allowed 30 times tol as in the parity tests.
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


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("n,nrhs", [(16, 1), (24, 9), (64, 33), (66, 3), (80, 32), (126, 65), (250, 8)])
def test_dense_lu_and_solve_at_tile_edges(pm, n, nrhs):
    prob = wl.star_grid(1, 1, n=n, seed=3, k_out=3.0)
    angs = list(np.linspace(0.1, 6.0, nrhs))
    x = pm.Factor(pm.Geometry(prob), 1e-12).solve(pm.Geometry(prob).plane_wave(angs))
    assert _rel(x, dense.solve(prob, angs)) < 1e-10


@pytest.mark.parametrize("nx,ny,n", [(2, 1, 80), (2, 2, 78), (3, 1, 96), (2, 2, 98), (3, 2, 130)])
def test_compressed_solution_at_panel_edges(pm, nx, ny, n):
    prob = wl.star_grid(nx, ny, n=n, seed=5, k_out=5.0)
    angs = [0.3, 2.1]
    g = pm.Geometry(prob)
    f = pm.Factor(g, 1e-12)
    plain = pm.Factor(g, 1e-12, qr_first=False)
    ref = dense.solve(prob, angs)
    F = g.plane_wave(angs)
    assert _rel(f.solve(F), ref) < 3e-11
    assert _rel(plain.solve(F), ref) < 3e-11
    # the reduction preserves the pivoted factorization: the same ranks up to a rank decision at its threshold
    assert abs(f.stats()["K"] - plain.stats()["K"]) <= 2 * nx * ny
