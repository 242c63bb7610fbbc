"""The grid-wide Jacobi PCG's general table on both sides of the row count from which it takes
two CTAs per SM (500,000): weighted chains, u and v side, both precisions.

Tolerance: a solve to 1e-12 in k iterations leaves a residual b - A x within 1e-12 |b| and the
rounding that k updates and the residual's own products carry, 4 (k + 10) u ||A| |x|| with
u = 2^-53."""
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


@pytest.mark.parametrize("prec", ["CR_FP64", "CR_MIXED"])
@pytest.mark.parametrize("n", [499999, 500000, 500003])
def test_weighted_chain(cr, n, prec):
    w = 0.5 + np.random.default_rng(n).random(n - 1)
    L = sp.diags([-w, np.r_[w, 0.0] + np.r_[0.0, w], -w], [-1, 0, 1], format="csr")
    Lc = synth.CSR(n, L.indptr.astype(np.int32), L.indices.astype(np.int32), L.data)
    rng = np.random.default_rng(1)
    X, Y = np.zeros((n, 2)), rng.standard_normal((n, 2))
    for a in range(2):
        X[n // 3 + 1000 * a: n // 3 + 1000 * a + 1500, a] = rng.random(1500)
    Om = (rng.random((n, 2)) > 0.25).astype(np.uint8)
    u, v = synth.random_unit(n, 1), synth.random_unit(n, 2)
    bu, bv = rng.standard_normal(n), rng.standard_normal(n)
    with cr.ConReg(Lc, Lc, X, Y, Om, 2.0, r_cap=1, pcg_tol=1e-12, pcg_maxit=5000, precision=getattr(cr, prec)) as g:
        (xu, ku), (xv, kv) = g.cr_solve_u(v, bu)[:2], g.cr_solve_v(u, bv)[:2]
        st = g.cr_get_stats()
    assert st["pcg_cluster"] == [0, 0] and st["pcg_multigrid"] == [0, 0], st
    om, s = Om @ (X.T @ v) ** 2, Om.T @ (u * u)
    for x, k, b, t, data in ((np.asarray(xu), ku, bu, v, lambda x: om * x),
                             (np.asarray(xv), kv, bv, u, lambda x: X @ (s * (X.T @ x)))):
        c, d = t @ (L @ t), np.sum((L @ t) ** 2)

        def apply(M, x):
            return 2.0 * (M @ (M @ x) + 2 * c * (M @ x) + d * x) + data(x)

        r, mag = b - apply(L, x), apply(abs(L), np.abs(x))
        assert np.linalg.norm(r) <= 1e-12 * np.linalg.norm(b) + 4 * (k + 10) * 2.0 ** -53 * np.linalg.norm(mag)
