"""The grid-wide Jacobi PCG with both of its neighbour tables (16-bit distances for
unit-weight graphs of near neighbours, 32-bit indices for the rest): sizes around
the four rows of a vector load, blocks without rows, weights, more than six
neighbours, a diagonal that is not the neighbour count; and inner products on
both sides of the two-stage limit.

Tolerance: solves to a relative residual of 1e-13 against a dense float64 solve,
20 cond 1.1e-13, at least 1e-9, as for the other PCG kernels."""
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


def graph(side, kind):
    n = side * side
    A = np.zeros((n, n))
    rng = np.random.default_rng(1)
    for y in range(side):
        for x in range(side):
            for dy, dx in [(0, 1), (1, 0)] + ([(1, 1), (1, -1)] if kind == "eight" else []):
                yy, xx = y + dy, x + dx
                if 0 <= yy < side and 0 <= xx < side:
                    w = rng.uniform(0.5, 1.5) if kind == "weighted" else 1.0
                    A[y * side + x, yy * side + xx] = A[yy * side + xx, y * side + x] = w
    L = np.diag(A.sum(1) + (0.25 if kind == "shifted" else 0.0)) - A
    r, c = np.nonzero(L)
    return synth.CSR(n, np.searchsorted(r, np.arange(n + 1)).astype(np.int32), c.astype(np.int32), L[r, c])


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("side,kind", [(7, "unit"), (10, "unit"), (13, "unit"), (9, "weighted"), (9, "eight"),
                                       (9, "shifted")])
def test_grid_pcg_tables(cr, side, kind, prec):
    p = synth.toy2d(side=side, m=3)
    L = graph(side, kind)
    p = dataclasses.replace(p, Lx=L, Ly=L)
    o = Oracle.from_problem(p)
    rng = np.random.default_rng(2)
    v, u = synth.random_unit(p.nx, 3), synth.random_unit(p.ny, 4)
    bu, bv = rng.standard_normal(p.ny), rng.standard_normal(p.nx)
    with cr.ConReg.from_problem(p, r_cap=2, pcg_tol=1e-13, pcg_maxit=50000, pcg_kernel=2,
                                precision=cr.CR_FP64 if prec == "fp64" else cr.CR_MIXED) as g:
        xu, xv = g.cr_solve_u(v, bu)[0], g.cr_solve_v(u, bv)[0]
        assert g.cr_get_stats()["pcg_cluster"] == [0, 0]
        assert np.array_equal(xu, g.cr_solve_u(v, bu)[0])
    Bs, s = o.B_hat(u)
    for x, A, b in ((xu, o.A_hat(v).toarray(), bu), (xv, Bs.toarray() + (p.X * s) @ p.X.T, bv)):
        ref = np.linalg.solve(A, b)
        assert np.linalg.norm(x - ref) <= max(1e-9, 20.0 * np.linalg.cond(A) * 1.1e-13) * np.linalg.norm(ref)


@pytest.mark.parametrize("n", [32768, 32769, 40001])
def test_long_inner_products(cr, n):
    """c = v' L v of a chain enters u_hat's system: with X = 0 it is lam (L^2 + 2 c L + d I) u = b."""
    rp = np.minimum(np.maximum(3 * np.arange(n + 1) - 1, 0), 3 * n - 2).astype(np.int32)
    i = np.arange(n)
    cols = np.stack([i - 1, i, i + 1], 1).ravel()
    vals = np.stack([-np.ones(n), np.full(n, 2.0), -np.ones(n)], 1)
    vals[0, 1] = vals[-1, 1] = 1.0
    keep = (cols >= 0) & (cols < n)
    L = synth.CSR(n, rp, cols[keep].astype(np.int32), vals.ravel()[keep])
    X, Y = np.zeros((n, 1)), np.zeros((n, 1))
    X[0, 0] = 1e-30  # a source that the system does not feel
    v = synth.random_unit(n, 1)
    b = np.random.default_rng(2).standard_normal(n)
    with cr.ConReg(L, L, X, Y, np.ones((n, 1), np.uint8), 1.0, r_cap=1, pcg_tol=1e-13) as g:
        x = g.cr_solve_u(v, b)[0]
    lap = lambda w: np.convolve(w, [-1.0, 2.0, -1.0], "same") - np.concatenate([w[:1], np.zeros(n - 2), w[-1:]])  # noqa: E731
    lv = lap(v)
    r = b - (lap(lap(x)) + 2.0 * (v @ lv) * lap(x) + (lv @ lv) * x)
    assert np.linalg.norm(r) <= 1e-11 * np.linalg.norm(b)  # c and d to a few 1e-16, |A| / lambda_min < 40
