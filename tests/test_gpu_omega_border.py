"""G_a = U^T diag(Omega_a) U kept up to date from the shorter of each injection's
row lists (cr_basis.cu): masks without observed or unobserved rows, with one of
them, exactly half, and both sorts in one problem.

Tolerance: the read-back is float32, so 1.2e-7 of each entry, and 1e-13 for the
float64 sums of products of orthonormal columns."""
import dataclasses

import numpy as np
import pytest

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


@pytest.mark.parametrize("shape,j", [((3, 2), 1), ((8, 4), 7), ((9, 7), 33), ((24, 20), 40)])
def test_galerkin_blocks(cr, shape, j):
    n = shape[0] * shape[1]
    p = synth.rect2d(shape_y=shape, shape_x=(8, 8), m=8)
    rng = np.random.default_rng(n)
    Om = np.zeros((n, 8), np.uint8)
    Om[:, 1] = 1
    Om[n // 2, 2] = 1
    Om[:, 3] = 1
    Om[n - 1, 3] = 0
    Om[: n // 2, 4] = 1
    Om[:, 5] = rng.random(n) < 0.3
    Om[:, 6] = rng.random(n) < 0.7
    Om[: n // 2 + 1, 7] = 1
    p = dataclasses.replace(p, Omega=Om)
    U, V = (np.linalg.qr(rng.standard_normal((k, j)))[0] for k in (n, 64))
    with cr.ConReg.from_problem(p, r_cap=j, precision=cr.CR_MIXED) as g:
        g.cr_set_factors(U, np.eye(j), V)
        G = g.cr_galerkin_assembly(1).astype(np.float64)
    ref = np.einsum("ia,ip,iq->apq", Om.astype(np.float64), U, U)
    assert np.all(np.abs(G - ref) <= 1.2e-7 * np.abs(ref) + 1e-13)
