"""The backward error of results that are not finite (needs a GB300): no
solution of NaN passes as converged, and right-hand sides that are not finite
themselves are taken as before.
"""
import numpy as np
import pytest

import oracle
from wdgen import Kernel, compressed_pattern, compressed_values, haar_basis, rhs

pytestmark = pytest.mark.gpu


def _one(scale=1.0):
    b = haar_basis(2, 4)
    cp, ri = compressed_pattern(b)
    return b, cp, ri, scale * compressed_values(b, cp, ri, Kernel("matern32", 0.1), 1e-3)


def _solver(wdlib, batch, scale=1.0):
    """(handle, n, values) of one system, or of three as a batch."""
    b, cp, ri, v = _one(scale)
    if not batch:
        return wdlib.Solver().analyze(cp, ri, b), b.N, v
    return wdlib.Solver().analyze_batch([(cp, ri)] * 3, [b] * 3), 3 * b.N, np.concatenate([v] * 3)


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("ncols", [1, 8, 9, 70])
def test_mixed_result_not_finite_is_an_error(wdlib, cuda, batch, ncols):
    """A finite right-hand side that FP32 cannot hold."""
    s, n, v = _solver(wdlib, batch)
    s.factor(v, "mixed")
    B = rhs(n, ncols, seed=1)
    B[:, -1] *= 1e200
    with pytest.raises(wdlib.WdError) as e:
        s.solve(B)
    assert e.value.status == wdlib.WD_ERR_NO_CONVERGENCE
    s.solve(rhs(n, ncols, seed=1))


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("ncols", [1, 8, 9, 70])
def test_fp64_result_not_finite_is_reported(wdlib, cuda, batch, ncols):
    s, n, v = _solver(wdlib, batch, 1e-200)
    s.factor(v, "fp64")
    B = rhs(n, ncols, seed=1)
    B[:, -1] *= 1e200
    s.solve(B)
    assert s.last_solve["backward_error"] == np.inf


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("ncols", [1, 8, 9, 70])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_backward_error_of_given_values(wdlib, cuda, batch, ncols, value):
    s, n, v = _solver(wdlib, batch)
    s.factor(v, "fp64")
    B = rhs(n, ncols, seed=2)
    X = s.solve(B)
    assert s.backward_error(X, B) <= 1e-12
    Y = X.copy()
    Y[n // 2, -1] = value
    assert s.backward_error(Y, B) == np.inf
    C = B.copy()
    C[n // 2, -1] = value           # no finite solution: the column does not count
    assert s.backward_error(X, C) <= 1e-12


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("ncols", [2, 8, 9, 70])
def test_right_hand_side_not_finite_is_taken(wdlib, cuda, prec, ncols):
    b, cp, ri, v = _one()
    s = wdlib.Solver().analyze(cp, ri, b).factor(v, prec)
    B = rhs(b.N, ncols, seed=3)
    B[5, 1] = np.nan
    X = s.solve(B)
    assert np.isnan(X[:, 1]).any()
    keep = np.arange(ncols) != 1
    assert oracle.backward_error(cp, ri, v, X[:, keep], B[:, keep]).max() <= 1e-12


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("ncols", [8, 9, 70])
@pytest.mark.parametrize("scale", [1e50, 1e-300])
def test_backward_error_beyond_fp32(wdlib, cuda, batch, ncols, scale):
    """Values that FP64 holds and FP32 does not: the residual of more than 8
    columns takes FP64 where double-float arithmetic overflows (1e50; 1e-300
    vanishes in it)."""
    s, n, v = _solver(wdlib, batch)
    s.factor(v, "fp64")
    B = scale * rhs(n, ncols, seed=4)
    X = s.solve(B)
    if scale > 1.0 or ncols <= 8:
        assert s.last_solve["backward_error"] <= 1e-12
        assert s.backward_error(X, B) <= 1e-12
    assert np.isfinite(X).all()
    for i in range(0, n, _one()[0].N):
        b, cp, ri, one = _one()
        assert oracle.backward_error(cp, ri, one, X[i:i + b.N], B[i:i + b.N]).max() <= 1e-12
