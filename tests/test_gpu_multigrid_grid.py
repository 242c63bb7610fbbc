"""The grid-wide multigrid PCG (cr_mg_grid.cu) where its row split, transfers and
tables can go wrong: two-level hierarchies, CTAs without rows, weighted
Laplacians and rows of more than six neighbours (no unit-weight path), source
and target grids of different sizes, the v side with and without the Woodbury
step (m on both sides of 32), against a dense float64 solve.

Tolerance: both sides solve to a relative residual of 1e-13, so the solutions
agree to cond(A) (1e-13 + n eps); 20 cond 1.1e-13, at least 1e-9, as for the
cluster kernel."""
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


def weighted(grid, seed, diagonals=False):
    """Graph Laplacian of a 2-D box with random edge weights; with diagonals, the 8-neighbour graph."""
    h, w = grid.mask.shape
    n = h * w
    rng = np.random.default_rng(seed)
    A = np.zeros((n, n))
    steps = [(0, 1), (1, 0)] + ([(1, 1), (1, -1)] if diagonals else [])
    for y in range(h):
        for x in range(w):
            for dy, dx in steps:
                yy, xx = y + dy, x + dx
                if 0 <= yy < h and 0 <= xx < w:
                    A[y * w + x, yy * w + xx] = A[yy * w + xx, y * w + x] = rng.uniform(0.5, 1.5)
    L = np.diag(A.sum(1)) - A
    r, c = np.nonzero(L)
    rp = np.searchsorted(r, np.arange(n + 1)).astype(np.int32)
    return synth.CSR(n, rp, c.astype(np.int32), L[r, c])


def problem(name):
    if name == "chain66":  # two rows more than the coarsest level may hold
        return synth.paper_toy(n=66, m=3)
    if name == "ragged":  # 23 x 29 and 21 x 31: different grids, CTAs with one row less
        return synth.rect2d(shape_y=(23, 29), shape_x=(21, 31), m=5, lam=20.0)
    if name == "m40":  # more injections than the Woodbury step takes
        return synth.toy2d(side=24, m=40)
    p = synth.toy2d(side=21, m=4)
    L = weighted(p.grid_x, 3, diagonals=name == "eight")
    return dataclasses.replace(p, Lx=L, Ly=L)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", ["chain66", "ragged", "m40", "weighted", "eight"])
def test_grid_multigrid_matches_dense_solve(cr, name, prec):
    p = problem(name)
    o = Oracle.from_problem(p)
    rng = np.random.default_rng(7)
    v, u = synth.smooth_unit(p.grid_x, 5), synth.smooth_unit(p.grid_y, 6)
    bu, bv = rng.standard_normal(p.ny), rng.standard_normal(p.nx)
    with cr.ConReg.from_problem(p, r_cap=2, pcg_tol=1e-13, pcg_maxit=200000,
                                precision=cr.CR_FP64 if prec == "fp64" else cr.CR_MIXED,
                                precond=cr.CR_PRECOND_MULTIGRID) as g:
        first = g.cr_solve_u(v, bu)[0], g.cr_solve_v(u, bv)[0]
        again = g.cr_solve_u(v, bu)[0], g.cr_solve_v(u, bv)[0]
        st = g.cr_get_stats()
    assert min(st["pcg_multigrid"]) >= 2 and st["pcg_cluster"] == [0, 0], st
    Bs, s = o.B_hat(u)
    for x, y, A, b in ((first[0], again[0], o.A_hat(v).toarray(), bu),
                       (first[1], again[1], Bs.toarray() + (p.X * s) @ p.X.T, bv)):
        ref = np.linalg.solve(A, b)
        bar = max(1e-9, 20.0 * np.linalg.cond(A) * 1.1e-13)
        assert np.linalg.norm(x - ref) <= bar * np.linalg.norm(ref)
        assert np.array_equal(x, y)  # fixed summation order
