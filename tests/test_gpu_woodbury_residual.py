"""The residual that a v-side multigrid solve with the Woodbury step reports is the
residual that its solution has, also at tolerances near float64's limit: the
recurrence's A u has to come from the u that enters x.

Tolerance: the solution's residual b - A x, formed in extended precision, is at most
three times the larger of the tolerance and what the one-cluster kernel
(cluster_size = 16), which runs the same recurrence in another summation order,
leaves."""
import numpy as np
import pytest

from paper_1808_05510_gb300 import synth

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def cr():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1808_05510_gb300 import build, conreg

    build.build()
    conreg.load()
    return conreg


def lap(L, x):
    return np.add.reduceat(L.val.astype(LD) * x[L.col], L.rowptr[:-1].astype(np.int64))


def true_residual(p, u, x, b):
    u, x, X = u.astype(LD), x.astype(LD), p.X.astype(LD)
    lu = lap(p.Ly, u)
    s = p.Omega.astype(LD).T @ (u * u)
    lx = lap(p.Lx, x)
    r = b - (LD(p.lam) * (lap(p.Lx, lx) + 2 * (u @ lu) * lx + (lu @ lu) * x) + X @ (s * (X.T @ x)))
    return float(np.linalg.norm(r) / np.linalg.norm(b.astype(LD)))


@pytest.mark.parametrize("m", [5, 28, 32])
@pytest.mark.parametrize("lam", [1.0, 30.0, 300.0])
def test_reported_residual_is_the_solutions(cr, lam, m):
    p = synth.visual_cortex(box=30, n_target=3000, m=m, lam=lam)
    u = synth.smooth_unit(p.grid_y, 6)
    b = (p.Y * p.Omega).T @ u
    b = p.X @ b
    left = {}
    for cs in (0, 16):
        with cr.ConReg.from_problem(p, r_cap=1, pcg_tol=1e-13, pcg_maxit=2000, precond=cr.CR_PRECOND_MULTIGRID,
                                    cluster_size=cs) as g:
            x = np.asarray(g.cr_solve_v(u, b)[0])
            st = g.cr_get_stats()
        assert st["pcg_multigrid"][1] >= 2 and (st["pcg_cluster"][1] == 0) == (cs == 0), st
        left[cs] = true_residual(p, u, x, b)
    print(lam, m, left)
    assert left[0] <= 3 * max(1e-13, left[16]), left
