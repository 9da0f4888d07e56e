"""Performance cases: what a user of the solver has it do, through its public entry points.

A case names a compressed operator (`family`, `n` unknowns), what is asked of it (`kind`), the
precision or option, and the number of right-hand sides.  The operators are the generators' own
(Haar wavelets, a = 2 compression): `line` (1D, exponential kernel), `square` (2D, Matern-3/2),
`square12` (2D, Matern-1/2, the gradient experiment), `square_ns` (2D with an antisymmetric
transport term), `sphere` (six patches, exponential kernel on the chordal distance) and `mixture`
(a batch of independent 1D and 2D instances).  `line` and `square` take any n: the finest level
is kept on a strip of the domain only (a locally refined basis), which is a principal submatrix
of the full operator, so sizes are ragged as well as powers of two.

The seed sets the variance of the kernel (the scale of the matrix without its nugget) and the
right-hand sides; patterns and the unit-variance matrices depend on the sizes alone.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2007_01541_gb300 as wd
from paper_2007_01541_gb300.autograd import SPDSystem, gp_negative_log_likelihood
from wdgen import (Basis, Kernel, batch_instances, compressed_pattern, compressed_values, fwt, haar_basis,
                   mass_matrix)
from wdgen.sphere import sphere_basis, sphere_pattern, sphere_values

DEV = "cuda"
KERNELS = {"line": Kernel("exponential", 0.2), "square": Kernel("matern32", 0.1),
           "square12": Kernel("matern12", 0.15), "square_ns": Kernel("exponential", 0.2),
           "sphere": Kernel("exponential", 0.3)}
NUGGETS = {"line": 1e-2, "square": 1e-3, "square12": 1e-2, "square_ns": 1e-2, "sphere": 1e-2}
TRANSPORT = 0.5         # weight of square_ns's antisymmetric term
THETA, DT = 0.5, 1e-2   # Crank-Nicolson


def listed():
    return [
        # The smallest call: a 1D Gaussian process with one data vector, host arrays in and out.
        dict(name="line_1024_fp64_host_1", kind="factor_solve", family="line", n=1024, prec="fp64", nrhs=1, host=True),
        # The headline workload: a new matrix is factored and 64 systems are solved to 1e-12.
        dict(name="square_65536_mixed_64", kind="factor_solve", family="square", n=65536, prec="mixed", nrhs=64),
        # One right-hand side against a kept factor: what a Krylov or Newton loop calls again and again.
        dict(name="square_65536_mixed_solve_1", kind="solve", family="square", n=65536, prec="mixed", nrhs=1),
        # The same matrix in full FP64, with the option that a user takes for large FP64 fronts.
        dict(name="square_65536_fp64tc_64", kind="factor_solve", family="square", n=65536, prec="fp64tc", nrhs=64),
        # Many right-hand sides against a kept FP64 factor (posterior variances), an uneven number.
        dict(name="square_16384_fp64_solve_130", kind="solve", family="square", n=16384, prec="fp64", nrhs=130),
        # A locally refined basis with an odd number of unknowns and of right-hand sides.
        dict(name="square_11003_mixed_33", kind="factor_solve", family="square", n=11003, prec="mixed", nrhs=33),
        # Forward and backward of the likelihood with 32 observation vectors (hyperparameter training).
        dict(name="square12_16384_grad_32", kind="grad", family="square12", n=16384, prec="fp64", nrhs=32),
        # Time stepping with one factor: 16 Crank-Nicolson steps of one state with a source.
        dict(name="square_16384_theta_1", kind="theta", family="square", n=16384, prec="mixed", nrhs=1, steps=16,
             mass=False),
        # Gaussian random field samples on the sphere: factor, then 128 samples P^T L z.
        dict(name="sphere_24576_sample_128", kind="sample", family="sphere", n=24576, prec="fp64", nrhs=128),
        # Many small independent systems of different sizes in one call, one right-hand side each.
        dict(name="mixture_64_mixed_1", kind="batch", family="mixture", count=64, pick=0, prec="mixed", nrhs=1),
        # A nonsymmetric operator (double layer): LU, 16 right-hand sides, log |det|.
        dict(name="square_ns_16384_lu_16", kind="lu", family="square_ns", n=16384, prec="lu", nrhs=16),
        # A symmetric indefinite operator: LDL^T, solves, log |det| and the inertia.
        dict(name="sphere_6144_ldlt_8", kind="ldlt", family="sphere", n=6144, prec="lu", nrhs=8),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["factor_solve"] * 5 + ["solve"] * 2 + ["theta", "sample", "batch", "grad", "lu", "ldlt"])
    if kind == "batch":
        return dict(kind=kind, family="mixture", count=log_int(3, 64), pick=rng.randrange(1, 1000),
                    prec=rng.choice(["mixed", "fp64"]), nrhs=rng.choice([1, 1, 2, 5]))
    if kind == "sample":
        return dict(kind=kind, family="sphere", n=rng.choice([1536, 6144, 24576]), prec="fp64", nrhs=log_int(1, 128))
    if kind == "ldlt":
        return dict(kind=kind, family="sphere", n=rng.choice([1536, 6144]), prec="lu", nrhs=log_int(1, 40))
    if kind == "lu":
        return dict(kind=kind, family="square_ns", n=rng.choice([1024, 4096, 16384]), prec="lu", nrhs=log_int(1, 40))
    if kind == "grad":
        return dict(kind=kind, family="square12", n=log_int(700, 16384), prec="fp64", nrhs=log_int(1, 48))
    if kind == "theta":
        return dict(kind=kind, family="square", n=log_int(700, 16384), prec="mixed", nrhs=rng.choice([1, 1, 3, 12]),
                    steps=rng.choice([4, 9, 16]), mass=rng.random() < 0.4)
    prec = rng.choice(["mixed", "mixed", "fp64", "fp64tc"])
    family = rng.choice(["square", "square", "line"])
    top = 16384 if family == "line" or prec == "fp64" else 65536
    return dict(kind=kind, family=family, n=log_int(300, top), prec=prec, nrhs=log_int(1, 64 if top > 16384 else 130))


# ---- inputs -----------------------------------------------------------------------------------
class _System:
    """Pattern, geometry and unit-variance values (without the nugget) of one operator."""

    def __init__(self, basis, colptr, rowidx, lower, upper=None, nugget=0.0):
        self.basis, self.colptr, self.rowidx, self.nugget = basis, colptr, rowidx, nugget
        self.lower = torch.as_tensor(lower, dtype=torch.float64, device=DEV)
        self.upper = None if upper is None else torch.as_tensor(upper, dtype=torch.float64, device=DEV)
        self.n = colptr.size - 1
        self.diag = torch.as_tensor(colptr[:-1], device=DEV)

    def values(self, scale, v=None):
        v = (self.lower if v is None else v) * scale
        v[self.diag] += self.nugget
        return v

    @functools.cached_property
    def mass(self):
        return torch.as_tensor(mass_matrix(self.basis, self.colptr, self.rowidx), device=DEV)


def _nonsymmetric_values(basis, colptr, rowidx, kernel):
    """wdgen.compressed_values_nonsym's matrix, formed on the GPU."""
    n, N = basis.n_side, basis.N
    c = (torch.arange(n, dtype=torch.float64, device=DEV) + 0.5) / n
    y, x = (t.reshape(-1) for t in torch.meshgrid(c, c, indexing="ij"))
    r = torch.sqrt((x[:, None] - x[None, :]).square_() + (y[:, None] - y[None, :]).square_())
    k = kernel(r, torch) * (1.0 + TRANSPORT * (x[:, None] - x[None, :]) / kernel.ell) / N
    del r
    k = fwt(k.reshape(N, n, n), 2, basis.J, torch)
    a = fwt(k.T.contiguous().reshape(N, n, n), 2, basis.J, torch).T     # T K T^T
    rows = torch.as_tensor(rowidx.astype(np.int64), device=DEV)
    cols = torch.repeat_interleave(torch.arange(N, device=DEV), torch.as_tensor(np.diff(colptr), device=DEV))
    return a[rows, cols].clone(), a[cols, rows].clone()


@functools.lru_cache(maxsize=None)
def _full(family, J):
    if family == "sphere":
        b = sphere_basis(J)
        cp, ri = sphere_pattern(b, DEV)
        sysm = _System(b, cp, ri, sphere_values(b, cp, ri, KERNELS[family], 0.0, DEV), nugget=NUGGETS[family])
    else:
        b = haar_basis(1 if family == "line" else 2, J)
        cp, ri = compressed_pattern(b)
        if family == "square_ns":
            sysm = _System(b, cp, ri, *_nonsymmetric_values(b, cp, ri, KERNELS[family]), nugget=NUGGETS[family])
        else:
            v = compressed_values(b, cp, ri, KERNELS[family], 0.0, DEV)
            sysm = _System(b, cp, ri, v, nugget=NUGGETS[family])
    torch.cuda.empty_cache()    # the dense kernel matrix
    return sysm


@functools.lru_cache(maxsize=None)
def _system(family, n):
    if family == "sphere":
        return _full(family, round(math.log(n // 6, 4)))
    dim = 1 if family == "line" else 2
    J = max(1, math.ceil(math.log2(n) / dim - 1e-9))
    full = _full(family, J)
    if full.n == n:
        return full
    b = full.basis
    fine = np.flatnonzero(b.level == J)
    keep = b.level < J
    keep[fine[np.argsort(b.box_lo[fine, 0], kind="stable")][:n - int(keep.sum())]] = True
    cols = np.repeat(np.arange(full.n), np.diff(full.colptr))
    sel = keep[cols] & keep[full.rowidx]
    new = np.cumsum(keep) - 1
    colptr = np.concatenate([[0], np.cumsum(np.bincount(new[cols[sel]], minlength=n))]).astype(np.int64)
    basis = Basis(b.dim, b.J, b.level[keep], b.box_lo[keep], b.box_side[keep])
    pick = torch.as_tensor(np.flatnonzero(sel), device=DEV)
    return _System(basis, colptr, new[full.rowidx[sel]].astype(np.int32), full.lower[pick], nugget=full.nugget)


@functools.lru_cache(maxsize=None)
def _mixture(count, pick):
    return [_system("line" if p["dim"] == 1 else "square12", p["N"]) for p in batch_instances(count, pick)]


def _options(case):
    return dict(fp64_tc_schur=True) if case["prec"] == "fp64tc" else {}


def _inputs(case, seed):
    """The numbers that the seed sets: values and right-hand sides (and the start and source of a step)."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(rng.integers(1 << 62)))

    def block(n):
        return torch.randn((case["nrhs"], n), dtype=torch.float64, device=DEV, generator=gen)

    if case["kind"] == "batch":
        systems = _mixture(case["count"], case["pick"])
        values = torch.cat([s.values(rng.uniform(0.5, 1.0)) for s in systems])
        return dict(values=values, B=block(sum(s.n for s in systems)))
    sysm = _system(case["family"], case["n"])
    scale = rng.uniform(0.5, 1.0)
    if case["kind"] == "lu":
        return dict(lower=sysm.values(scale), upper=sysm.values(scale, sysm.upper), B=block(sysm.n))
    if case["kind"] == "ldlt":
        # the nugget of 1e-3 leaves the compressed matrix indefinite
        values = sysm.lower * (2.0 * scale)
        values[sysm.diag] += 1e-3
        return dict(values=values, B=block(sysm.n))
    values = sysm.values(scale)
    if case["kind"] == "theta":
        mass = sysm.mass if case["mass"] else torch.zeros_like(values).index_fill_(0, sysm.diag, 1.0)
        return dict(values=mass + THETA * DT * values, operator=values, mass=mass if case["mass"] else None,
                    B=block(sysm.n), F=block(sysm.n))
    return dict(values=values, B=block(sysm.n))


def prepare(case, seed):
    state = _inputs(case, seed)
    state["case"] = case
    kind = case["kind"]
    if kind == "grad":
        sysm = _system(case["family"], case["n"])
        state["system"] = SPDSystem(sysm.colptr, sysm.rowidx, sysm.basis)
        state["values"].requires_grad_(True)
        state["B"].requires_grad_(True)
        return state
    solver = state["solver"] = wd.Solver(**_options(case))
    if kind == "batch":
        systems = _mixture(case["count"], case["pick"])
        solver.analyze_batch([(s.colptr, s.rowidx) for s in systems], [s.basis for s in systems])
    else:
        sysm = _system(case["family"], case["n"])
        solver.analyze(sysm.colptr, sysm.rowidx, sysm.basis)
    if case.get("host"):
        state["values"] = state["values"].cpu().numpy()
        state["B"] = state["B"].cpu().numpy().T
    if kind in ("solve", "theta"):
        solver.factor(state["values"], _precision(case))
    if kind == "theta" and state["mass"] is not None:
        solver.set_mass(state["mass"])
    return state


def _precision(case):
    return "mixed" if case["prec"] == "mixed" else "fp64"


def run(state):
    case = state["case"]
    kind, B = case["kind"], state["B"]
    if kind == "grad":
        loss = gp_negative_log_likelihood(state["system"], state["values"], B.t())
        gvalues, gB = torch.autograd.grad(loss, (state["values"], B))
        return dict(loss=loss.detach(), gvalues=gvalues, gB=gB)
    s = state["solver"]
    if kind in ("factor_solve", "batch"):
        s.factor(state["values"], _precision(case))
    if kind in ("factor_solve", "solve", "batch"):
        X = s.solve(B) if case.get("host") else s.solve(B.clone().t())
        # the mixed factor is FP32, and so would its log det be: it is asked of FP64 factors
        if case["prec"] == "mixed" or kind == "solve":
            return dict(X=X)
        return dict(X=X, logdet=s.logdet_batch() if kind == "batch" else s.logdet())
    if kind == "theta":
        U = B.clone().t()
        F = state["F"].t()
        for _ in range(case["steps"]):
            s.theta_step(U, F, THETA, DT)
        return dict(U=U)
    if kind == "sample":
        s.factor(state["values"], "fp64")
        return dict(S=s.apply_L(B.t()))
    if kind == "lu":
        s.factor_lu(state["lower"], state["upper"])
        X = s.solve_lu(B.clone().t())
        logabs, sign = s.logdet_lu()
        return dict(X=X, logabs=logabs, sign=sign)
    s.factor_ldlt(state["values"])
    X = s.solve_lu(B.clone().t())
    logabs, sign = s.logdet_lu()
    npos, nneg = s.inertia()
    return dict(X=X, logabs=logabs, sign=sign, npos=npos, nneg=nneg)


# ---- what a pass cannot do without -----------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _counts(family, n):
    """(entries of A stored, entries of L, factorization flops) of the default ordering."""
    sysm = _system(family, n)
    s = wd.Solver(symbolic_only=True).analyze(sysm.colptr, sysm.rowidx, sysm.basis)
    i = s.info()
    s.close()
    return i["nnz_A_lower"], i["nnz_L"], i["flops_factor"]


def work(case):
    kind, r = case["kind"], case["nrhs"]
    if kind == "batch":
        sizes = [(s.n, _counts("line" if s.basis.dim == 1 else "square12", s.n)) for s in _mixture(case["count"], case["pick"])]
        n = sum(x for x, _ in sizes)
        nnz, nl, fl = (sum(c[q] for _, c in sizes) for q in range(3))
    else:
        n = case["n"]
        nnz, nl, fl = _counts(case["family"], n)
    item = 4 if case["prec"] == "mixed" else 8
    vectors = 16 * n * r                     # read once, written once
    if kind in ("factor_solve", "batch"):
        return dict(bytes=8 * nnz + vectors, flops=fl + 4.0 * nl * r)
    if kind == "solve":
        return dict(bytes=item * nl + vectors, flops=4.0 * nl * r)
    if kind == "theta":
        # per step: the factor once, the matrix (and the mass matrix) once
        m = 2 if case["mass"] else 1
        return dict(bytes=case["steps"] * (item * nl + 8 * m * nnz + 1.5 * vectors),
                    flops=case["steps"] * (4.0 * nl + 4.0 * m * nnz) * r)
    if kind == "sample":
        return dict(bytes=8 * nnz + vectors, flops=fl + 2.0 * nl * r)
    if kind == "grad":
        # factor, two solves, the selected inverse (twice the factor's flops), the gradient's outer products
        return dict(bytes=16 * nnz + 2 * vectors, flops=3 * fl + 8.0 * nl * r + 4.0 * nnz * r)
    both = 2 if kind == "lu" else 1
    return dict(bytes=8 * both * nnz + vectors, flops=2 * fl + 4.0 * nl * r)


# ---- the same in 64 bits by dense algebra ------------------------------------------------------------
def _indices(sysm):
    rows = torch.as_tensor(sysm.rowidx.astype(np.int64), device=DEV)
    cols = torch.repeat_interleave(torch.arange(sysm.n, device=DEV), torch.as_tensor(np.diff(sysm.colptr), device=DEV))
    return rows, cols


def _dense(sysm, lower, upper=None):
    rows, cols = _indices(sysm)
    A = torch.zeros((sysm.n, sysm.n), dtype=torch.float64, device=DEV)
    A[cols, rows] = lower if upper is None else upper
    A[rows, cols] = lower
    return A


def _spd_solve(A, B):
    """(X, log det) by Cholesky and one step of refinement."""
    C = torch.linalg.cholesky(A)
    X = torch.cholesky_solve(B, C)
    X += torch.cholesky_solve(B - A @ X, C)
    return X, 2.0 * torch.log(torch.diagonal(C)).sum()


def _cg(sysm, values, B, tol=1e-15, most=2000):
    """Conjugate gradients on all columns at once, for matrices too large for the dense factor."""
    rows, cols = _indices(sysm)
    off = rows != cols
    idx = torch.cat([torch.stack([rows, cols]), torch.stack([cols[off], rows[off]])], 1)
    A = torch.sparse_coo_tensor(idx, torch.cat([values, values[off]]), (sysm.n, sysm.n)).coalesce().to_sparse_csr()
    X = torch.zeros_like(B)
    for _ in range(2):                      # the second time on the true residual
        R = B - A @ X
        P, rho, D, start = R.clone(), R.square().sum(0), torch.zeros_like(B), R.square().sum(0)
        for _ in range(most):
            Q = A @ P
            alpha = rho / (P * Q).sum(0).clamp_min(1e-300)
            D += alpha * P
            R -= alpha * Q
            new = R.square().sum(0)
            if bool((new <= tol * tol * start).all()):
                break
            P = R + (new / rho.clamp_min(1e-300)) * P
            rho = new
        X += D
    return X


def exact(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    B = x["B"].t()
    if kind == "batch":
        out, dets, n0, e0 = [], [], 0, 0
        for s in _mixture(case["count"], case["pick"]):
            X, ld = _spd_solve(_dense(s, x["values"][e0:e0 + s.rowidx.size]), B[n0:n0 + s.n])
            out.append(X)
            dets.append(float(ld))
            n0, e0 = n0 + s.n, e0 + s.rowidx.size
        X = torch.cat(out)
        return dict(X=X) if case["prec"] == "mixed" else dict(X=X, logdet=np.array(dets))
    sysm = _system(case["family"], case["n"])
    if kind in ("factor_solve", "solve"):
        if sysm.n > 24576:
            X, ld = _cg(sysm, x["values"], B), None
        else:
            X, ld = _spd_solve(_dense(sysm, x["values"]), B)
            ld = float(ld)
        if case.get("host"):
            X = X.cpu().numpy()
        return dict(X=X) if case["prec"] == "mixed" or kind == "solve" else dict(X=X, logdet=ld)
    if kind == "theta":
        K = _dense(sysm, x["operator"])
        G = torch.eye(sysm.n, dtype=torch.float64, device=DEV) if x["mass"] is None else _dense(sysm, x["mass"])
        C = torch.linalg.cholesky(G + THETA * DT * K)
        G -= (1.0 - THETA) * DT * K
        U, F = B, x["F"].t()
        for _ in range(case["steps"]):
            U = torch.cholesky_solve(G @ U + DT * F, C)
        return dict(U=U)
    if kind == "sample":
        # the elimination order is the solver's own choice: it is taken from it, the numbers are not
        s = wd.Solver(symbolic_only=True).analyze(sysm.colptr, sysm.rowidx, sysm.basis)
        perm = torch.as_tensor(s.symbolic()["perm"].astype(np.int64), device=DEV)
        s.close()
        A = _dense(sysm, x["values"])[perm][:, perm]
        S = torch.empty((B.shape[1], sysm.n), dtype=torch.float64, device=DEV).t()
        S[perm] = torch.linalg.cholesky(A) @ B
        return dict(S=S)
    if kind == "grad":
        A = _dense(sysm, x["values"])
        X, ld = _spd_solve(A, B)
        Z = torch.cholesky_inverse(torch.linalg.cholesky(A))
        rows, cols = _indices(sysm)
        w = torch.where(rows == cols, 1.0, 2.0).to(torch.float64)
        m = B.shape[1]
        gv = 0.5 * m * w * Z[rows, cols]
        for c in range(m):                  # d/dv of 1/2 b^T A^-1 b is -1/2 x x^T
            gv -= 0.5 * w * X[rows, c] * X[cols, c]
        return dict(loss=0.5 * (B * X).sum() + 0.5 * m * ld, gvalues=gv, gB=X.t())
    A = _dense(sysm, x["lower"], x["upper"]) if kind == "lu" else _dense(sysm, x["values"])
    LU, piv = torch.linalg.lu_factor(A)
    X = torch.linalg.lu_solve(LU, piv, B)
    X += torch.linalg.lu_solve(LU, piv, B - A @ X)
    out = dict(X=X, logabs=float(torch.log(torch.abs(torch.diagonal(LU))).sum()), sign=None)
    return out if kind == "lu" else dict(out, npos=None, nneg=None)
