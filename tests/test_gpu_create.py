"""What a problem's creation computes, on the host and on the device: the basis of X's columns
(zero, repeated and dependent ones are left out) and |D|_F from it, and one set-up
for two equal Laplacians.

Tolerance: ||R|| / ||D|| against the dense oracle to 1e-10 relative, the bound of
the residual tests; solves to a relative residual of 1e-13 against a dense float64
solve, 20 cond 1.1e-13, at least 1e-9, as for the other PCG kernels."""
import dataclasses

import numpy as np
import pytest

from oracle import Oracle
from paper_1808_05510_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cr():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1808_05510_gb300 import build, conreg

    build.build()
    conreg.load()
    return conreg


# the basis is made on the host up to m max(nx, ny) = 25,000
@pytest.mark.parametrize("shape", [(6, 8), (64, 65), (64, 66)])
@pytest.mark.parametrize("kind", ["plain", "zero", "repeated", "dependent", "allzero"])
def test_basis_of_x(cr, kind, shape):
    p = synth.rect2d(shape_y=(9, 7), shape_x=shape, m=6)
    X = p.X.copy()
    if kind == "zero":
        X[:, [0, 3]] = 0.0
    elif kind == "repeated":
        X[:, 4] = X[:, 1]
    elif kind == "dependent":
        X[:, 5] = 0.5 * X[:, 0] - 2.0 * X[:, 2]
    elif kind == "allzero":
        X[:] = 0.0
    p = dataclasses.replace(p, X=X)
    if kind == "allzero":  # no column at all: accepted
        with cr.ConReg.from_problem(p, r_cap=4) as g:
            assert g.cr_get_rank() == 0
        return
    o = Oracle.from_problem(p)
    rng = np.random.default_rng(3)
    U, V = (np.linalg.qr(rng.standard_normal((n, 4)))[0] for n in (p.ny, p.nx))
    Z = rng.standard_normal((4, 4))
    R, D = np.linalg.norm(o.D() - o.A_op(U @ Z @ V.T)), np.linalg.norm(o.D())
    with cr.ConReg.from_problem(p, r_cap=4) as g:
        assert abs(g.cr_residual()["relres"] - 1.0) <= 1e-10  # no factors yet: R = D
        g.cr_set_factors(U, Z, V)
        got = g.cr_residual()["relres"]
    assert abs(got - R / D) <= 1e-10 * R / D


def scaled(L, f):
    return synth.CSR(L.n, L.rowptr.copy(), L.col.copy(), L.val * f)


@pytest.mark.parametrize("precond", ["CR_PRECOND_JACOBI", "CR_PRECOND_MULTIGRID"])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("kind", ["copy", "scaled", "other"])
def test_equal_and_unequal_grids(cr, kind, prec, precond):
    p = synth.toy2d(side=20, m=3)
    Ly = scaled(p.Lx, 1.0 if kind == "copy" else 2.0)
    if kind == "other":
        Ly = synth.rect2d(shape_y=(40, 10), shape_x=(6, 8), m=2).Ly  # the same number of rows
    p = dataclasses.replace(p, Ly=Ly)
    o = Oracle.from_problem(p)
    rng = np.random.default_rng(2)
    v, u = synth.random_unit(p.nx, 3), synth.random_unit(p.ny, 4)
    bu, bv = rng.standard_normal(p.ny), rng.standard_normal(p.nx)
    with cr.ConReg.from_problem(p, r_cap=2, pcg_tol=1e-13, pcg_maxit=50000, precond=getattr(cr, precond),
                                precision=cr.CR_FP64 if prec == "fp64" else cr.CR_MIXED) as g:
        xu, xv = np.asarray(g.cr_solve_u(v, bu)[0]), np.asarray(g.cr_solve_v(u, bv)[0])
    Bs, sc = o.B_hat(u)
    for x, A, b in ((xu, o.A_hat(v).toarray(), bu), (xv, Bs.toarray() + (p.X * sc) @ p.X.T, bv)):
        ref = np.linalg.solve(A, b)
        assert np.linalg.norm(x - ref) <= max(1e-9, 20.0 * np.linalg.cond(A) * 1.1e-13) * np.linalg.norm(ref)
