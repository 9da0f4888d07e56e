"""FP64 pivots over the whole range of exponents (needs a GB300): quotients by
reciprocals and, near and beyond the ends of the normal range, by division.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _lower_csc(A):
    n = A.shape[0]
    cp = np.concatenate([[0], np.cumsum(np.arange(n, 0, -1))]).astype(np.int64)
    ri = np.concatenate([np.arange(j, n) for j in range(n)]).astype(np.int32)
    return cp, ri, np.concatenate([A[j:, j] for j in range(n)])


def _scaled(n, p, exponent):
    """S positive definite with unit diagonal; A = D S D with unknown p scaled
    to a pivot of about 2^exponent."""
    M = np.random.default_rng(n).standard_normal((n, n))
    S = M @ M.T + n * np.eye(n)
    S /= np.sqrt(np.outer(np.diag(S), np.diag(S)))
    D = np.ones(n)
    D[p] = 2.0 ** (exponent / 2)
    A = S * D[:, None] * D
    A[p, p] = S[p, p] * 2.0 ** exponent       # D[p]^2 in one rounding
    return S, D, A


# 2^-1030 keeps 44 bits, and p > 0 subtracts from it: columns to 1e-11
@pytest.mark.parametrize("exponent", [-1030, -1022, -1002, -1000, -998, 998, 1000, 1002, 1020])
@pytest.mark.parametrize("n,p", [(20, 0), (20, 5), (70, 0), (70, 63), (70, 66), (130, 70)])
@pytest.mark.parametrize("kind", ["fp64", "ldlt", "lu"])
def test_factor_with_an_extreme_pivot(wdlib, cuda, kind, n, p, exponent):
    if kind == "lu" and n > 64:
        pytest.skip("L's panels multiply by inverses of U11, which overflow")
    S, D, A = _scaled(n, p, exponent)
    cp, ri, v = _lower_csc(A)
    C = np.linalg.cholesky(S)
    s = wdlib.Solver().analyze(cp, ri)
    if kind == "fp64":
        got, ref = [s.factor(v, "fp64").L_csc_like(cp, ri)], [D[:, None] * C]
    else:
        s.factor_ldlt(v) if kind == "ldlt" else s.factor_lu(v, v)
        got = [s.L_csc_like(cp, ri, x) for x in s.export_LU()]
        c = np.diag(C)
        with np.errstate(over="ignore"):
            ref = [D[:, None] * (C / c) / D, D[:, None] * (C * c) * D]
    col, row = np.repeat(np.arange(n), np.arange(n, 0, -1)), ri
    for g, r in zip(got, ref):
        want = r[row, col]
        assert np.isfinite(want).all() and np.isfinite(g).all()
        for j in range(n):
            e = col == j
            # per column, past the scale of row p
            w = np.where(row[e] == p, 1.0 / D[p], 1.0)
            sc = 1.0 / np.abs(want[e] * w).max()
            assert np.abs(((g[e] - want[e]) * w) * sc).max() <= 1e-11, j


def test_quotients_are_rounded_like_divisions(wdlib, cuda):
    """L21 = w / d of 2 x 2 blocks, d of every exponent and either sign, within
    one unit in the last place."""
    rng = np.random.default_rng(0)
    e = np.repeat(np.arange(-1070, 1023), 3)
    cnt = e.size
    d = np.ldexp(rng.uniform(1.0, 2.0, cnt), e) * rng.choice([-1.0, 1.0], cnt)
    w = d * rng.uniform(0.25, 0.5, cnt)
    keep = w != 0.0
    d, w, cnt = d[keep], w[keep], int(keep.sum())
    cp = np.concatenate([[0], np.cumsum(np.tile([2, 1], cnt))]).astype(np.int64)
    ri = (2 * np.repeat(np.arange(cnt), 3) + np.tile([0, 1, 1], cnt)).astype(np.int32)
    lower = np.stack([d, w, np.ones(cnt)], 1).reshape(-1)
    upper = np.stack([d, np.zeros(cnt), np.ones(cnt)], 1).reshape(-1)
    s = wdlib.Solver(relax_k=0, relax_pct=0).analyze(cp, ri).factor_lu(lower, upper)
    L = s.L_csc_like(cp, ri, s.export_LU()[0]).reshape(cnt, 3)[:, 1]
    q = w / d
    assert (np.abs(L - q) <= np.spacing(np.abs(q))).all()
