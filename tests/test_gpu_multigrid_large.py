"""The grid-wide multigrid PCG with its tables in device memory (cr_mg_grid.cu): above some
60,000 rows they no longer fit the CTAs' shared memory.  u and v side, both precisions, with
and without the Woodbury step.

Tolerance: a solve to 1e-11 in k iterations leaves a residual b - A x within 1e-11 |b| and the
rounding that k updates of x and r and the residual's own products carry, 4 (k + 10) u times
||A| |x|| with u = 2^-53."""
import numpy as np
import pytest
import scipy.sparse as sp

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


def problem(m):
    rng = np.random.default_rng(m)
    g = synth.Grid(synth.shell_mask((120, 80, 100), 80000))
    L = synth.grid_laplacian(g)
    X = synth.gaussian_injections(g, m, rng, 2.0, 3.0, 0.2, 1.0)
    return g, L, X, rng.random((g.n, m)), (X < 1e-3).astype(np.uint8)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("m", [8, 40])
def test_tables_in_device_memory(cr, m, prec):
    grid, Lc, X, Y, Om = problem(m)
    n, lam = grid.n, 1e3
    assert 70000 <= n <= 110000
    u, v = synth.smooth_unit(grid, 6), synth.smooth_unit(grid, 5)
    D = Y * Om
    with cr.ConReg(Lc, Lc, X, Y, Om, lam, r_cap=1, pcg_tol=1e-11, pcg_maxit=2000, precond=cr.CR_PRECOND_MULTIGRID,
                   precision=cr.CR_FP64 if prec == "fp64" else cr.CR_MIXED) as g:
        bu, bv = D @ (X.T @ v), X @ (D.T @ u)
        (xu, ku), (xv, kv) = g.cr_solve_u(v, bu)[:2], g.cr_solve_v(u, bv)[:2]
        st = g.cr_get_stats()
    assert min(st["pcg_multigrid"]) >= 2 and st["pcg_cluster"] == [0, 0], st
    L = sp.csr_matrix((Lc.val, Lc.col, Lc.rowptr), shape=(n, n))
    om, s = Om @ (X.T @ v) ** 2, Om.T @ (u * u)
    for x, k, b, w, data in ((np.asarray(xu), ku, bu, v, lambda x: om * x),
                             (np.asarray(xv), kv, bv, u, lambda x: X @ (s * (X.T @ x)))):
        c, d = w @ (L @ w), np.sum((L @ w) ** 2)

        def apply(M, x):
            return lam * (M @ (M @ x) + 2 * c * (M @ x) + d * x) + data(x)

        r, mag = b - apply(L, x), apply(abs(L), np.abs(x))
        assert np.linalg.norm(r) <= 1e-11 * np.linalg.norm(b) + 4 * (k + 10) * 2.0 ** -53 * np.linalg.norm(mag)
