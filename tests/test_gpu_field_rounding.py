"""Rounding error of the field sums over many nodes.

Reference: the far field of the same node data and boundary values in extended
precision.  Yardstick: a float64 restatement that adds every node's finished
term to a thread's sum, 64 nodes a thread here.  In units of a term's variance
its running sums contribute sum_{i<=64} i = 2,080; the library's runs of eight
nodes 8 x 68 within the runs and 8 x 36 between them, 832; fused
multiply-adds straight into the running sum would contribute 4,128.  What both
have in common (sine, cosine, the products of a term) brings the ratios nearer
to one, not across it.
"""
import numpy as np
import pytest

from paper_2603_09381_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _far(ld, k, x, n, w, q, u, ang):
    """terms (direction, node), complex in the type ld, without the factor in front"""
    k = ld(k)
    x, n, w = x.astype(ld), n.astype(ld), w.astype(ld)
    ca, sa = np.cos(ang.astype(ld))[:, None], np.sin(ang.astype(ld))[:, None]
    ph = -k * (ca * x[:, 0] + sa * x[:, 1])
    kn = k * (ca * n[:, 0] + sa * n[:, 1])
    s, c = np.sin(ph), np.cos(ph)
    tx = kn * u.imag.astype(ld) - q.real.astype(ld)
    ty = -kn * u.real.astype(ld) - q.imag.astype(ld)
    return w * (c * tx - s * ty), w * (c * ty + s * tx)


def _block_sum(t):
    """the library's order: 256 threads, node i in thread i % 256; lanes pairwise, then the warps in turn"""
    a = np.zeros((t.shape[0], 256))
    for m in range(t.shape[1] // 256):
        a = a + t[:, 256 * m:256 * (m + 1)]
    a = a.reshape(-1, 8, 32)
    while a.shape[2] > 1:
        h = a.shape[2] // 2
        a = a[:, :, :h] + a[:, :, h:]
    out = np.zeros(t.shape[0])
    for wp in range(8):
        out = out + a[:, wp, 0]
    return out


def test_far_field_rounding_stays_below_that_of_finished_terms():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_09381_gb300 import pmchwt as pm
    k = 0.5
    prob = wl.circle_grid(2, 2, n=4096, k_out=k, k_in=1.0)
    g = pm.Geometry(prob)
    x, nrm, w = g.nodes()
    rng = np.random.default_rng(5)
    phi = rng.standard_normal((g.N, 2)) + 1j * rng.standard_normal((g.N, 2))
    ang = np.linspace(0.05, 6.2, 48)
    got = g.far_field(phi, ang)
    gm = 0.25 * np.sqrt(2.0 / (np.pi * k)) * np.sqrt(0.5)   # e^{i pi/4} / sqrt(2) x sqrt(2)
    err, yard = [], []
    for c in range(phi.shape[1]):
        blocks = phi[:, c].reshape(4, 2, 4096)
        q, u = blocks[:, 0].ravel(), blocks[:, 1].ravel()
        ex = [np.sum(t, axis=1) for t in _far(np.longdouble, k, x, nrm, w, q, u, ang)]
        f64 = [_block_sum(t) for t in _far(np.float64, k, x, nrm, w, q, u, ang)]
        # out = gm ((tx - ty) + i (tx + ty)); the library's sums from its outputs, the factor's rounding well below theirs
        z = got[:, c] / gm
        lib = [(z.real + z.imag) / 2, (z.imag - z.real) / 2]
        for p in range(2):
            err.append(lib[p] - ex[p].astype(np.longdouble))
            yard.append(f64[p] - ex[p])
    rms = lambda v: float(np.sqrt(np.mean(np.square(np.array(v, dtype=np.longdouble)))))
    print("rms error", rms(err), "yardstick", rms(yard))
    assert rms(err) < rms(yard)
