"""R_j v and R_j^T u with factors of every rank around a warp's edge: the operator's
coefficient rows are summed by a warp each (cr_small.cu).

Tolerance: 1e-12 of the result, the bound of the residual product tests (sums of
the same terms in another order)."""
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


@pytest.mark.parametrize("j", [1, 2, 3, 5, 31, 32, 33, 48])
def test_residual_products(cr, j):
    p = synth.rect2d(shape_y=(9, 7), shape_x=(6, 8), m=4)
    o = Oracle.from_problem(p)
    rng = np.random.default_rng(j)
    U, V = (np.linalg.qr(rng.standard_normal((n, j)))[0] for n in (p.ny, p.nx))
    Z = rng.standard_normal((j, j))  # not symmetric: a transposed one shows
    v, u = rng.standard_normal(p.nx), rng.standard_normal(p.ny)
    with cr.ConReg.from_problem(p, r_cap=min(j + 2, p.nx)) as g:
        g.cr_set_factors(U, Z, V)
        for got, want in ((g.cr_apply_residual(v), o.R_times(U, Z, V, v)),
                          (g.cr_apply_residual(u, trans=True), o.Rt_times(U, Z, V, u))):
            assert np.linalg.norm(got - want) <= 1e-12 * np.linalg.norm(want)
