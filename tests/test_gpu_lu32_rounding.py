"""Rounding of the complex64 LU that preconditions the refinement.

A single inclusion in the mixed mode is one dense complex64 LU, corrected once
per solve from the FP64 residual, so that the residual after the first
refinement step measures its backward error (squared).  Yardstick: the same step
with a complex64 elimination in panels of 32 columns that rounds every entry of
a panel at every column, restated here, and exact triangular solves.  Such an
LU on the device comes out at 1.5 times the yardstick, its solves round as
well; sums over groups of columns halve the squared error and stay below it.
"""
import ctypes as ct

import numpy as np
import pytest
import scipy.linalg as sl

from oracle import dense
from paper_2603_09381_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _fms(a, l, u):
    """a - l u, each component by two fused multiply-adds in FP32"""
    r32 = lambda v: v.astype(np.float32).astype(np.float64)
    p = [np.asarray(v, dtype=np.complex128) for v in (a, l, u)]
    (ar, ai), (lr, li), (ur, ui) = ((v.real, v.imag) for v in p)
    return (r32(r32(ar - lr * ur) + li * ui) + 1j * r32(r32(ai - lr * ui) - li * ur)).astype(np.complex64)


def _lu_by_columns(A, nb=32):
    A, n = A.astype(np.complex64), len(A)
    perm = np.arange(n)
    for p in range(0, n, nb):
        e = min(n, p + nb)
        for c in range(p, e):
            piv = c + int(np.argmax(np.abs(A[c:, c])))
            if piv != c:
                A[[c, piv]], perm[[c, piv]] = A[[piv, c]], perm[[piv, c]]
            A[c + 1:, c] *= np.complex64(1) / A[c, c]
            A[c + 1:, c + 1:e] = _fms(A[c + 1:, c + 1:e], A[c + 1:, c, None], A[None, c, c + 1:e])
        for c in range(p, e):
            A[c + 1:e, e:] = _fms(A[c + 1:e, e:], A[c + 1:e, c, None], A[None, c, e:])
        acc = np.zeros((n - e, n - e), np.complex64)
        for c in range(p, e):
            acc = _fms(acc, -A[e:, c, None], A[None, c, e:])
        A[e:, e:] -= acc
    return A, perm


def test_first_residual_stays_below_that_of_elimination_by_columns():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_09381_gb300 import pmchwt as pm
    got, yard = [], []
    for n in (114, 200):
        for seed in range(6):
            prob = wl.star_grid(1, 1, n=n, seed=seed, k_out=2.0 + seed)
            g = pm.Geometry(prob)
            b = g.plane_wave([0.3, 2.0, 4.1])
            f = pm.Factor(g, 1e-10, precision=pm.PM_MIXED, refine_tol=1e-14, max_refine=1)
            rhs = np.ascontiguousarray(b.T)
            out, info = np.zeros_like(rhs), pm.pm_solve_info()
            pm.load().pm_solve_ex(f.h, rhs.ctypes.data, 3, out.ctypes.data, 0, ct.byref(info))   # (not converged)
            got.append(info.history[0])
            A = dense.assemble(prob)
            F, perm = _lu_by_columns(A)
            L, U = np.tril(F, -1).astype(complex) + np.eye(2 * n), np.triu(F).astype(complex)
            S = lambda v: sl.solve_triangular(U, sl.solve_triangular(L, v[perm], lower=True, unit_diagonal=True))
            x = S(b).astype(np.complex64).astype(complex)
            x = x + S(b - A @ x).astype(np.complex64)
            yard.append(np.max(np.linalg.norm(b - A @ x, axis=0) / np.linalg.norm(b, axis=0)))
    mean = lambda v: float(np.exp(np.mean(np.log(v))))
    print("first residual", mean(got), "yardstick", mean(yard))
    assert mean(got) < mean(yard)
