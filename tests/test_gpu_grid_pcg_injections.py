"""The grid-wide Jacobi PCG (cr_pcg_grid.cu) with the injections of whole data sets and
with as many as a problem takes: the v side's y = s o X^T p lies in dynamic shared
memory beside the kernel's own.

Tolerance: solves to a relative residual of 1e-13 against a dense float64 solve,
20 cond 1.1e-13, at least 1e-9, as for the other PCG kernels."""
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


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("m", [126, 1000, 4096])
def test_many_injections(cr, m, prec):
    p = synth.rect2d(shape_y=(9, 11), shape_x=(10, 13), m=m, lam=20.0)
    o = Oracle.from_problem(p)
    rng = np.random.default_rng(2)
    v, u = synth.random_unit(p.nx, 3), synth.random_unit(p.ny, 4)
    bu, bv = rng.standard_normal(p.ny), rng.standard_normal(p.nx)
    with cr.ConReg.from_problem(p, r_cap=2, pcg_tol=1e-13, pcg_maxit=50000, pcg_kernel=2,
                                precision=cr.CR_FP64 if prec == "fp64" else cr.CR_MIXED) as g:
        xu, xv = g.cr_solve_u(v, bu)[0], g.cr_solve_v(u, bv)[0]
        assert g.cr_get_stats()["pcg_cluster"] == [0, 0]
    Bs, s = o.B_hat(u)
    for x, A, b in ((xu, o.A_hat(v).toarray(), bu), (xv, Bs.toarray() + (p.X * s) @ p.X.T, bv)):
        ref = np.linalg.solve(A, b)
        assert np.linalg.norm(x - ref) <= max(1e-9, 20.0 * np.linalg.cond(A) * 1.1e-13) * np.linalg.norm(ref)
