"""G_a = U^T diag(Omega_a) U (cr_basis.cu) where most of a column's mass lies in the rows that
injection a does not observe, so that the observed rows' sum is far below u_p^T u_q.

Tolerance: the read-back is float32, 1.2e-7 of each entry; with u = 2^-53, a float64 sum of n
products is within n u of the sum of their absolute values over the observed rows.  Taken as
the difference from u_p^T u_q the sum also carries the unobserved rows' rounding, which is
accepted up to once the size of the result: 4 n u in all."""
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


@pytest.mark.parametrize("shape,j,decay", [((8, 4), 5, 1e-3), ((9, 7), 33, 1e-6), ((24, 20), 20, 1e-9), ((24, 20), 4, 0.0)])
def test_blocks_to_the_size_of_the_observed_sum(cr, shape, j, decay):
    n = shape[0] * shape[1]
    p = synth.rect2d(shape_y=shape, shape_x=(8, 8), m=4)
    rng = np.random.default_rng(n + j)
    Om = np.ones((n, 4), np.uint8)
    hidden = rng.permutation(n)[: n // 3]
    Om[hidden, 0] = 0          # the mass of every column
    Om[hidden[::2], 1] = 0     # half of it
    Om[:, 2] = 0
    Om[hidden, 2] = 1          # the same rows as observed ones: the short list holds them
    p = dataclasses.replace(p, Omega=Om)
    U = rng.standard_normal((n, j))
    U[np.setdiff1d(np.arange(n), hidden)] *= decay
    U /= np.linalg.norm(U, axis=0)
    V = np.linalg.qr(rng.standard_normal((64, j)))[0]
    with cr.ConReg.from_problem(p, r_cap=j, precision=cr.CR_MIXED) as g:
        g.cr_set_factors(U, np.eye(j), V)
        G = g.cr_galerkin_assembly(1).astype(np.float64)
    Ul, O = U.astype(np.longdouble), Om.astype(np.longdouble)
    ref = np.einsum("ia,ip,iq->apq", O, Ul, Ul)
    mag = np.einsum("ia,ip,iq->apq", O, np.abs(Ul), np.abs(Ul))
    assert np.all(np.abs(G - ref) <= 1.2e-7 * np.abs(ref) + 4 * n * 2.0 ** -53 * mag)
