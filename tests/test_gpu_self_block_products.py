"""Self blocks as the factorizations assemble them (Maue products on the tensor
cores at FP64 accuracy) against the oracle, at the edges of the products' 128 x
32 tiles and 32-term stages.

Entries agree to the rounding of the products: the differentiation matrix has
norm n / 2 and the single layer decays as 1 / |m| over the modes, so that the
error is about n 2^-53 of the block, below 1e-12 at 258 nodes with a wide margin.
"""
import numpy as np
import pytest

from oracle import blocks, geometry
from paper_2603_09381_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16, 34, 62, 96, 126, 130, 258])
@pytest.mark.parametrize("lossy", [False, True])
def test_self_block_matches_oracle_at_tile_edges(n, lossy):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_09381_gb300 import pmchwt as pm
    prob = wl.star_grid(1, 1, n=n, seed=2, k_out=3.0)
    if lossy:
        prob["inclusions"][0]["k_in"] *= 1 + 0.05j
    nd = geometry.all_nodes(prob)[0]
    inc = prob["inclusions"][0]
    A = pm.Geometry(prob).self_block(0, n)
    ref = blocks.self_block(nd, prob["k_out"], inc["k_in"], 1.0, geometry.eps_in(prob, 0))
    assert np.linalg.norm(A - ref) < 1e-12 * np.linalg.norm(ref)
