"""The field sums on both sides of one run of eight nodes a thread (2,048 nodes
in 256 threads): the totals are kept above it only.

Reference: the oracle's formulas on the same boundary values.  Tolerance: both
sum N terms with a relative error of a few eps each, the oracle pairwise, the
library over at most N / 256 + 13 levels; random values make the sum about
sqrt(N) times smaller than the sum of the moduli.  (N / 256 + 13 + 30) eps
sqrt(N) is below 6e-13 at the largest N here, Hankel arguments' reduction
included; 2e-12 is asked.
"""
import numpy as np
import pytest

from oracle import field
from paper_2603_09381_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,n", [(1, 1, 2046), (8, 4, 64), (5, 5, 82), (1, 2, 2048), (1, 2, 2050)])
def test_field_sums_around_one_run(nx, ny, n):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_09381_gb300 import pmchwt as pm
    prob = wl.circle_grid(nx, ny, n=n)
    g = pm.Geometry(prob)
    rng = np.random.default_rng(n)
    phi = rng.standard_normal((g.N, 15)) + 1j * rng.standard_normal((g.N, 15))   # groups of 8, 4, 2, 1
    ang = np.linspace(0.1, 6.0, 5)
    pts = np.stack([np.linspace(-1, 7, 5), np.full(5, -3.0)], -1)
    ff, us = g.far_field(phi, ang), g.scattered_field(phi, pts)
    for c in (0, 7, 8, 11, 12, 13, 14):
        rf, ru = field.far_field(prob, phi[:, c], ang), field.scattered_field(prob, phi[:, c], pts)
        assert np.linalg.norm(ff[:, c] - rf) < 2e-12 * np.linalg.norm(rf)
        assert np.linalg.norm(us[:, c] - ru) < 2e-12 * np.linalg.norm(ru)
    np.testing.assert_array_equal(g.far_field(phi[:, :1], ang)[:, 0], ff[:, 0])   # (the same bits in any group)
    np.testing.assert_array_equal(g.scattered_field(phi[:, :1], pts)[:, 0], us[:, 0])
