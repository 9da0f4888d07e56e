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
