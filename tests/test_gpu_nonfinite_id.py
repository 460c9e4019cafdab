"""A complex128 ID input that is not finite is reported, not taken for zeros.

The pivoted QR holds its columns in fixed point, which has no NaN.  A NaN
written into the first ID input has to end the factorization, with the tall
input reduced to its triangle first (96 nodes: the NaN spreads to all later
columns of the panel) or pivoted on directly.
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


@pytest.mark.parametrize("n,qr_first,predicted", [(96, True, False), (96, False, False), (48, True, False), (48, True, True)])
def test_a_nan_in_an_id_input_is_reported(pm, n, qr_first, predicted):
    prob = wl.star_grid(2, 1, n=n, seed=1, k_out=3.0)
    kw = {}
    if predicted:
        from paper_2603_09381_gb300 import rank_predictor as rp
        dm = rp.to_device(rp.load_model())
        kw["rank_model"] = dm.data_ptr()
    g = pm.Geometry(prob)
    with pytest.raises(pm.PmError) as e:
        pm.Factor(g, 1e-10, qr_first=qr_first, debug_flags=pm.PM_DEBUG_NONFINITE_ID, **kw)
    assert e.value.status == 4 and "not finite" in str(e.value)
    x = pm.Factor(g, 1e-10, qr_first=qr_first, **kw).solve(g.plane_wave([0.5]))
    ref = dense.solve(prob, [0.5])
    assert np.linalg.norm(x - ref) < 1e-8 * np.linalg.norm(ref)
