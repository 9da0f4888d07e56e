"""Calls repeated after WD_ERR_OOM (needs a GB300; memory runs out on the host
side of the allocator): nothing half made is taken for ready.
"""
import numpy as np
import pytest

import oracle
from wdgen import Kernel, compressed_pattern, compressed_values, haar_basis, rhs

pytestmark = pytest.mark.gpu

_c = {}


def _small():
    if not _c:
        b = haar_basis(2, 5)
        cp, ri = compressed_pattern(b)
        _c.update(b=b, cp=cp, ri=ri, v=compressed_values(b, cp, ri, Kernel("matern32", 0.1), 1e-3))
    return _c["b"], _c["cp"], _c["ri"], _c["v"]


def _each_allocation(wdlib, call, **opts):
    """call(solver, attempt) with the k-th device allocation failing, for every
    k; attempt(f, ...) is f(...), done again if it ran out of memory."""
    failures = 0
    for k in range(1, 300):
        s = wdlib.Solver(test_fail_alloc=k, **opts)
        failed = []

        def attempt(f, *args, between=None):
            try:
                return f(*args)
            except wdlib.WdError as e:
                assert e.status == wdlib.WD_ERR_OOM, (k, str(e))
                failed.append(1)
                if between:
                    between()
                return f(*args)

        call(s, attempt)
        s.close()
        assert len(failed) <= 1
        failures += len(failed)
        if not failed:
            return failures
    pytest.fail("more than 299 device allocations")


def test_solve_of_another_kind(wdlib, cuda):
    """The same number of right-hand sides in another precision: the plan is
    made anew, and its buffers with it."""
    b, cp, ri, v = _small()
    B = rhs(b.N, 40, seed=0)

    def call(s, attempt):
        attempt(s.analyze, cp, ri, b)
        for prec in ("mixed", "fp64", "mixed"):
            attempt(s.factor, v, prec)
            X = attempt(s.solve, B)
            assert oracle.backward_error(cp, ri, v, X, B).max() <= 1e-12

    assert _each_allocation(wdlib, call) >= 10


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_fewer_columns_after_a_failed_solve(wdlib, cuda, prec):
    """A wider solve that runs out of memory gives the workspaces back; the
    next, narrower one makes its own."""
    b, cp, ri, v = _small()
    B = rhs(b.N, 70, seed=0)

    def call(s, attempt):
        attempt(s.analyze, cp, ri, b)
        attempt(s.factor, v, prec)

        def narrow():
            X = s.solve(B[:, :3])
            assert oracle.backward_error(cp, ri, v, X, B[:, :3]).max() <= 1e-12
            s.apply_L(B[:, :3])

        for c in (3, 40, 70):
            X = attempt(s.solve, B[:, :c], between=narrow)
            assert oracle.backward_error(cp, ri, v, X, B[:, :c]).max() <= 1e-12
            attempt(s.apply_L, B[:, :c], between=narrow)

    assert _each_allocation(wdlib, call) >= 10


def test_factor_with_slices(wdlib, cuda):
    """FP64 updates on the tensor cores: the slices' planes and their scales."""
    b, cp, ri, v = _small()
    B = rhs(b.N, 3, seed=0)

    def call(s, attempt):
        attempt(s.analyze, cp, ri, b)
        attempt(s.factor, v, "fp64")
        X = attempt(s.solve, B)
        assert oracle.backward_error(cp, ri, v, X, B).max() <= 1e-12

    assert _each_allocation(wdlib, call, fp64_tc_schur=True) >= 10


def test_selected_inverse_and_gradient(wdlib, cuda):
    """The pattern's maps are made by whichever call needs them first."""
    b, cp, ri, v = _small()
    U = rhs(b.N, 2, seed=0)
    col = np.repeat(np.arange(b.N), np.diff(cp))
    outer = 2.0 * (U[ri] * U[col]).sum(1) * np.where(ri == col, 0.5, 1.0)
    ref = wdlib.Solver().analyze(cp, ri, b).factor(v, "fp64").selinv()

    def call(s, attempt):
        attempt(s.analyze, cp, ri, b)
        assert np.abs(attempt(s.sym_pattern_outer, U, U) - outer).max() <= 1e-12 * np.abs(outer).max()
        attempt(s.factor, v, "fp64")
        np.testing.assert_array_equal(attempt(s.selinv), ref)
        assert np.abs(attempt(s.sym_pattern_outer, U, U) - outer).max() <= 1e-12 * np.abs(outer).max()

    assert _each_allocation(wdlib, call) >= 10


def test_level_schedule(wdlib, cuda):
    """A schedule that does not fit leaves the one before in place."""
    b, cp, ri, v = _small()
    B = rhs(b.N, 3, seed=0)

    def call(s, attempt):
        attempt(s.analyze, cp, ri, b)

        def solved():
            X = attempt(s.factor, v, "mixed").solve(B)
            assert oracle.backward_error(cp, ri, v, X, B).max() <= 1e-12

        attempt(s.factor, v, "mixed")
        attempt(s.solve, B)
        flags = [1] * len(s.level_schedule())

        def before():
            assert s.level_schedule() == [0] * len(flags)
            solved()

        attempt(s.set_level_schedule, flags, between=before)
        assert s.level_schedule() == flags
        solved()

    assert _each_allocation(wdlib, call) >= 10


@pytest.mark.parametrize("nrhs", [5, 16, 17, 130])
def test_lu_solve_takes_fewer_columns_at_a_time(wdlib, cuda, nrhs):
    """Where the workspaces of 64 columns do not fit those of 32 or 16 do: with
    more than 16 columns one allocation that fails does not fail the call."""
    b, cp, ri, v = _small()
    B = rhs(b.N, nrhs, seed=0)
    in_solve = []

    def call(s, attempt):
        attempt(s.analyze, cp, ri, b)
        attempt(s.factor_lu, v, v)

        def solve():
            try:
                return s.solve_lu(B)
            except wdlib.WdError:
                in_solve.append(1)
                raise

        assert oracle.backward_error(cp, ri, v, attempt(solve), B).max() <= 1e-12
        assert oracle.backward_error(cp, ri, v, attempt(solve), B).max() <= 1e-12

    _each_allocation(wdlib, call)
    assert (len(in_solve) == 0) == (nrhs > 16)
