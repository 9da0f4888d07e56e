"""One handle, several factorizations in turn (needs a GB300): the FP32 and
FP64 fronts share one pool, so what an earlier factor of any kind left there
must not reach the results of a later one.

The earlier factor is one of a matrix of NaN: every entry it stores is NaN in
its own type and, word by word, in the other one.  The kernels add in a fixed
order, so the later results are bit for bit those of a fresh handle.
"""
import numpy as np
import pytest

from wdgen import Kernel, compressed_pattern, compressed_values, haar_basis, rhs

pytestmark = pytest.mark.gpu


def _bordered(r, k=300):
    """Two dense blocks of k unknowns, each coupled to the same r: fronts of k
    pivot columns with r rows below (and 20 rows of padding between)."""
    rng = np.random.default_rng(r)
    n = 2 * k + r
    A = np.zeros((n, n))
    for c in range(2):
        M = rng.standard_normal((k, k))
        A[c * k:(c + 1) * k, c * k:(c + 1) * k] = M @ M.T + k * np.eye(k)
        A[2 * k:, c * k:(c + 1) * k] = 0.3 * rng.standard_normal((r, k))
    M = rng.standard_normal((r, r))
    A[2 * k:, 2 * k:] = M @ M.T + n * np.eye(r)
    A = np.tril(A)
    cp = np.concatenate([[0], np.cumsum((A != 0).sum(0))]).astype(np.int64)
    return cp, np.nonzero(A.T)[1].astype(np.int32), A.T[A.T != 0], None


def _tree(J):
    b = haar_basis(2, J)
    cp, ri = compressed_pattern(b)
    return cp, ri, compressed_values(b, cp, ri, Kernel("matern32", 0.1), 1e-3), b


CASES = {"r1": lambda: _bordered(1), "r2": lambda: _bordered(2), "r3": lambda: _bordered(3),
         "r5": lambda: _bordered(5), "tree32": lambda: _tree(5), "tree64": lambda: _tree(6)}
_made = {}


def _factor(wdlib, s, kind, v):
    """The factorization; a matrix of NaN may be refused, its factor is left all the same."""
    try:
        if kind == "lu":
            s.factor_lu(v, v)
        elif kind == "ldlt":
            s.factor_ldlt(v)
        else:
            s.factor(v, kind)
    except wdlib.WdError as e:
        assert np.isnan(v).all() and e.status == wdlib.WD_ERR_NOT_SPD


def _results(s, kind, n, ncols):
    B = rhs(n, ncols, seed=ncols)
    if kind in ("lu", "ldlt"):
        return [s.solve_lu(B), np.array(s.logdet_lu()), *s.export_LU()]
    out = [s.solve(B), np.array(s.logdet()), s.apply_L(B)]
    return out + [s.selinv()] if kind == "fp64" else out


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("later", ["mixed", "mixed_simt", "mixed_step", "fp64", "fp64_tc", "lu", "ldlt"])
def test_factor_after_another_kind(wdlib, cuda, name, later):
    if name not in _made:
        _made[name] = CASES[name]()
    cp, ri, v, basis = _made[name]
    opts = dict(relax_k=0, relax_pct=0) if basis is None else {}
    opts.update(dict(mixed_simt=dict(solve_simt=True), mixed_step=dict(step_launches=True),
                     fp64_tc=dict(fp64_tc_schur=True)).get(later, {}))
    kind = later.split("_")[0]
    n = cp.size - 1
    fresh = wdlib.Solver(**opts).analyze(cp, ri, basis)
    _factor(wdlib, fresh, kind, v)
    ref = {c: _results(fresh, kind, n, c) for c in (3, 9, 40, 64)}
    for r in ref.values():
        assert all(np.isfinite(x).all() for x in r)
    for earlier in ("fp64", "lu", "ldlt", "mixed"):
        s = wdlib.Solver(**opts).analyze(cp, ri, basis)
        _factor(wdlib, s, earlier, v * np.nan)
        _factor(wdlib, s, kind, v)
        for c, r in ref.items():
            for got, want in zip(_results(s, kind, n, c), r):
                np.testing.assert_array_equal(got, want, err_msg=f"{later} after {earlier}, {c} columns")


@pytest.mark.parametrize("kind", ["lu", "ldlt"])
def test_lu_keeps_one_front_pool(wdlib, cuda, kind):
    """U^T lies in the upper parts of L's fronts: next to a Cholesky factor's
    memory LU takes the values once more per triangle and U's block inverses,
    here an eighth of the fronts, and no second pool."""
    cp, ri, v, basis = _tree(7)

    def used(k):
        cuda.cuda.synchronize()
        before = cuda.cuda.mem_get_info()[0]
        s = wdlib.Solver().analyze(cp, ri, basis)
        _factor(wdlib, s, k, v)
        return before - cuda.cuda.mem_get_info()[0], s.info()["front_bytes"]

    used("fp64")                            # module loading
    chol, fronts = used("fp64")
    lu, _ = used(kind)
    assert fronts > 400 << 20
    assert lu - chol <= fronts / 4
