"""The tiled kernels at the edges of their tiles, against the CPU oracle
(needs a GB300).  Tolerances as in test_gpu_parity.py: FP64 results differ
from the oracle's by summation order only.
"""
import numpy as np
import pytest

import oracle
from wdgen import Kernel, compressed_pattern, compressed_values, haar_basis, rhs

pytestmark = pytest.mark.gpu

_cache = {}


def _case(dim, J):
    if (dim, J) not in _cache:
        b = haar_basis(dim, J)
        cp, ri = compressed_pattern(b)
        v = compressed_values(b, cp, ri, Kernel("exponential", 0.2), 1e-2)
        o = oracle.Oracle(cp, ri, b)
        assert o.factor(v) == 0
        _cache[dim, J] = (b, cp, ri, v, o)
    return _cache[dim, J]


@pytest.mark.parametrize("dim,J", [(1, 3), (2, 5)])
@pytest.mark.parametrize("ncols", [1, 7, 8, 9, 32, 33])
def test_apply_L_column_tiles(wdlib, cuda, dim, J, ncols):
    b, cp, ri, v, o = _case(dim, J)
    Z = rhs(o.n, ncols, seed=3)
    ref = o.apply_L(Z)
    s = wdlib.Solver().analyze(cp, ri, b)
    for prec, tol in (("fp64", 1e-12), ("mixed", 1e-5)):   # mixed: the FP32 factor
        assert np.abs(s.factor(v, prec).apply_L(Z) - ref).max() <= tol * np.abs(ref).max()


def _lower_csc(A):
    n = A.shape[0]
    cp = np.concatenate([[0], np.cumsum(np.arange(n, 0, -1))]).astype(np.int64)
    ri = np.concatenate([np.arange(j, n) for j in range(n)]).astype(np.int32)
    return cp, ri, np.concatenate([A[j:, j] for j in range(n)])


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 33, 48, 63, 64, 65, 97, 128, 131, 200])
def test_fp64_block_edges(wdlib, cuda, n):
    """One dense front: pivot blocks and update tiles cut at every remainder."""
    rng = np.random.default_rng(n)
    M = rng.standard_normal((n, n))
    A = M @ M.T + n * np.eye(n)
    cp, ri, v = _lower_csc(A)
    s = wdlib.Solver().analyze(cp, ri).factor(v, "fp64")
    L = np.zeros((n, n))
    L[np.concatenate([np.arange(j, n) for j in range(n)]), np.repeat(np.arange(n), np.arange(n, 0, -1))] = \
        s.L_csc_like(cp, ri)
    ref = np.linalg.cholesky(A)
    assert np.linalg.norm(L - ref, axis=0).max() <= 1e-12 * np.linalg.norm(ref)
    B = rhs(n, 3, seed=1)
    assert oracle.backward_error(cp, ri, v, s.solve(B), B).max() <= 1e-14


@pytest.mark.parametrize("bad", [0, 15, 16, 40, 63, 64, 99])
def test_fp64_pivot_status(wdlib, cuda, bad):
    n = 100
    A = np.eye(n) * 2.0 + 0.001
    A[bad, bad] = -1.0
    cp, ri, v = _lower_csc(A)
    s = wdlib.Solver().analyze(cp, ri)
    with pytest.raises(wdlib.WdError) as e:
        s.factor(v, "fp64")
    assert e.value.status == wdlib.WD_ERR_NOT_SPD and e.value.column == bad


@pytest.mark.parametrize("kind", ["lu", "ldlt"])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 33, 63, 64, 65, 97, 131, 200])
def test_lu_block_edges(wdlib, cuda, kind, n):
    """One dense front, nonsymmetric or symmetric indefinite, diagonally
    dominant (so that no pivot is small); per-column tolerance 1e-10 as in
    test_lu.py."""
    rng = np.random.default_rng(n)
    A = rng.standard_normal((n, n))
    if kind == "ldlt":
        A = A + A.T
    A += np.diag(np.where(rng.random(n) < 0.5, -2.0, 2.0) * n)
    cp, ri, lo = _lower_csc(A)
    up = _lower_csc(np.ascontiguousarray(A.T))[2]
    o = oracle.Oracle(cp, ri)
    assert o.factor_lu(lo, up) == 0
    s = wdlib.Solver().analyze(cp, ri)
    s.factor_lu(lo, up) if kind == "lu" else s.factor_ldlt(lo)
    for got, ref in zip(s.export_LU(), o.lu_values()):
        got = s.L_csc_like(o.Lp, o.Li, got)
        for j in range(n):
            a, e = o.Lp[j], o.Lp[j + 1]
            assert np.linalg.norm(got[a:e] - ref[a:e]) <= 1e-10 * np.linalg.norm(ref[a:e]), j
    assert s.logdet_lu()[1] == o.logdet_lu()[1]
    if kind == "ldlt":
        assert s.inertia()[1] == int((np.linalg.eigvalsh(A) < 0).sum())


@pytest.mark.parametrize("nrhs", [64, 65, 130])
def test_lu_solve_passes(wdlib, cuda, nrhs):
    """More right-hand sides than one pass takes: even and uneven passes."""
    rng = np.random.default_rng(nrhs)
    n = 150
    A = rng.standard_normal((n, n)) + np.diag(np.full(n, 2.0 * n))
    cp, ri, lo = _lower_csc(A)
    up = _lower_csc(np.ascontiguousarray(A.T))[2]
    s = wdlib.Solver().analyze(cp, ri).factor_lu(lo, up)
    B = rhs(n, nrhs, seed=0)
    for _ in range(2):                       # the second time with the kept plan
        X = s.solve_lu(B)
        assert oracle.nonsym_backward_error(cp, ri, lo, up, X, B).max() <= 1e-13


@pytest.mark.parametrize("opts", [dict(), dict(solve_simt=True)])
@pytest.mark.parametrize("nrhs", [9, 16, 17, 32, 33, 49])
def test_solve_tiles(wdlib, cuda, opts, nrhs):
    """The 32 x 32 tiles of the solves, split and not, in FP64 and (by option)
    FP32: a tree of fronts and one dense front wider than a super-block."""
    b, cp, ri, v, o = _case(2, 5)
    n = 600
    rng = np.random.default_rng(n)
    M = rng.standard_normal((n, n))
    dense = _lower_csc(M @ M.T + n * np.eye(n))
    prec = "mixed" if opts else "fp64"
    for c, r, vals, basis in ((cp, ri, v, b), dense + (None,)):
        B = rhs(c.size - 1, nrhs, seed=nrhs)
        s = wdlib.Solver(**opts).analyze(c, r, basis).factor(vals, prec)
        assert oracle.backward_error(c, r, vals, s.solve(B), B).max() <= 1e-12


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 8])
def test_narrow_solve_edges(wdlib, cuda, prec, nrhs):
    """Up to 8 right-hand sides: dense fronts around the widths of blocks and
    super-blocks, and trees with many children and rows below."""
    rng = np.random.default_rng(nrhs)
    cases = []
    for n in (1, 31, 33, 64, 511, 513, 600):
        M = rng.standard_normal((n, n))
        cases.append(_lower_csc(M @ M.T + n * np.eye(n)) + (None,))
    for dim, J in ((1, 3), (1, 9), (2, 5)):
        b, cp, ri, v, _ = _case(dim, J)
        cases.append((cp, ri, v, b))
    n = 70                                   # an arrow: 69 children of one root
    A = np.eye(n) * 4.0
    A[-1, :-1] = A[:-1, -1] = 0.3
    A[-1, -1] = n
    cp = np.arange(0, 2 * n, 2)
    cp = np.concatenate([cp, [2 * n - 1]]).astype(np.int64)
    ri = np.array([x for j in range(n - 1) for x in (j, n - 1)] + [n - 1], np.int32)
    cases.append((cp, ri, A[ri, np.repeat(np.arange(n), np.diff(cp))], None))
    for cp, ri, v, basis in cases:
        B = rhs(cp.size - 1, nrhs, seed=nrhs)
        s = wdlib.Solver(relax_k=0, relax_pct=0).analyze(cp, ri, basis).factor(v, prec)
        assert oracle.backward_error(cp, ri, v, s.solve(B), B).max() <= 1e-12


@pytest.mark.parametrize("ncols", [1, 3, 8, 9, 12, 32, 33, 64, 66, 130])
def test_residual_chunks(wdlib, cuda, ncols):
    """The residual products' rows and rows cut into chunks, through the
    backward error of a given X.  The residual's
    double-float arithmetic (about 48 bits) leaves the estimate within 5e-15
    of the FP64 one."""
    for dim, J in ((2, 5), (1, 9), (2, 2)):
        b, cp, ri, v, o = _case(dim, J)
        s = wdlib.Solver().analyze(cp, ri, b).factor(v, "fp64")
        rng = np.random.default_rng(ncols)
        B = rhs(o.n, ncols, seed=ncols)
        X = o.solve(B) * (1.0 + 1e-7 * rng.standard_normal(B.shape))
        ref = oracle.backward_error(cp, ri, v, X, B).max()
        assert abs(s.backward_error(X, B) - ref) <= 5e-15 + 1e-9 * ref


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("nrhs", [1, 2, 4, 8])
def test_narrow_solve_large_launches(wdlib, cuda, prec, nrhs):
    """Enough fronts in one level that its launches take the shallow form: 700
    small dense blocks, each coupled to the same three unknowns."""
    rng = np.random.default_rng(nrhs)
    k, cnt, b = 5, 700, 3
    n = k * cnt + b
    M = rng.standard_normal((cnt, k, k))
    A = M @ M.transpose(0, 2, 1) + k * np.eye(k)
    border = np.arange(k * cnt, n)
    rows, vals = [], []
    for c in range(cnt):
        for j in range(k):
            rows.append(np.concatenate([np.arange(c * k + j, (c + 1) * k), border]))
            vals.append(np.concatenate([A[c, j:, j], 0.3 * rng.standard_normal(b)]))
    for j in range(b):
        rows.append(border[j:])
        vals.append(np.concatenate([[float(n)], np.ones(b - 1 - j)]))
    cp = np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int64)
    ri, v = np.concatenate(rows).astype(np.int32), np.concatenate(vals)
    B = rhs(n, nrhs, seed=nrhs)
    s = wdlib.Solver(relax_k=0, relax_pct=0).analyze(cp, ri).factor(v, prec)
    assert oracle.backward_error(cp, ri, v, s.solve(B), B).max() <= 1e-12


@pytest.mark.parametrize("dim,J", [(2, 4), (2, 5)])
def test_solve_after_fp64_factor(wdlib, cuda, dim, J):
    """The FP64 factor leaves words in the shared front pool that are NaN as
    FP32 above the diagonals of a later mixed factor; a reduction that starts
    inside a super-block (its end no multiple of 32) must not see them."""
    b, cp, ri, v, o = _case(dim, J)
    B = rhs(o.n, 40, seed=5)
    s = wdlib.Solver().analyze(cp, ri, b)
    s.factor(v, "fp64")
    X = s.factor(v, "mixed").solve(B)
    assert oracle.backward_error(cp, ri, v, X, B).max() <= 1e-12


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("cnt", [1, 2, 4, 5, 6, 9, 10])
def test_extend_add_children(wdlib, cuda, prec, cnt):
    """A dense front of 140 unknowns (more than one slice of rows) with cnt - 1
    children, fewer and more than one group of them."""
    rng = np.random.default_rng(cnt)
    k, b = 7, 140
    n = k * cnt + b
    A = np.zeros((n, n))
    for c in range(cnt):
        M = rng.standard_normal((k, k))
        A[c * k:(c + 1) * k, c * k:(c + 1) * k] = M @ M.T + k * np.eye(k)
        A[k * cnt:, c * k:(c + 1) * k] = 0.3 * rng.standard_normal((b, k))
    M = rng.standard_normal((b, b))
    A[k * cnt:, k * cnt:] = M @ M.T + n * np.eye(b)
    A = np.tril(A)
    cp = np.concatenate([[0], np.cumsum((A != 0).sum(0))]).astype(np.int64)
    ri = np.nonzero(A.T)[1].astype(np.int32)
    v = A.T[A.T != 0]
    B = rhs(n, 3, seed=cnt)
    s = wdlib.Solver(relax_k=0, relax_pct=0).analyze(cp, ri).factor(v, prec)
    assert oracle.backward_error(cp, ri, v, s.solve(B), B).max() <= (1e-14 if prec == "fp64" else 1e-12)
