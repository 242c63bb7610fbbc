"""Growth of the residual-norm bases, three columns of both grids at a time
(cr_basis.cu): columns that depend on earlier ones or on one another (an
eigenvector's L-images, pairs that span the same two eigenvectors, a full basis),
grids of different sizes, blocks without rows, and more basis columns than one pass
of the projection takes (1,536).

Tolerance: ||R|| / ||D|| against the dense oracle to 1e-10 relative, the bound
of the residual tests: the bases are orthonormal to a few 1e-16, and the terms
that add up to R are at most some 1e3 times larger than it here."""
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


def eigvecs(L):
    A = np.zeros((L.n, L.n))
    for i in range(L.n):
        A[i, L.col[L.rowptr[i] : L.rowptr[i + 1]]] = L.val[L.rowptr[i] : L.rowptr[i + 1]]
    return np.linalg.eigh(A)[1]


def columns(E, j, kind):
    """j orthonormal columns; "span": pairs (e1 + e2, e1 - e2), whose L-images stay in one plane."""
    if kind == "eigen":
        return E[:, :j].copy()
    if kind == "span":
        U = np.empty((E.shape[0], j))
        for q in range(j):
            a, b = E[:, 2 * (q // 2)], E[:, 2 * (q // 2) + 1]
            U[:, q] = (a + b if q % 2 == 0 else a - b) / np.sqrt(2.0)
        return U
    return np.linalg.qr(np.random.default_rng(5).standard_normal((E.shape[0], j)))[0]


@pytest.mark.parametrize("kind", ["random", "eigen", "span"])
@pytest.mark.parametrize("sy,sx,j,m", [((2, 2), (3, 3), 4, 2), ((9, 7), (3, 2), 6, 3), ((5, 5), (20, 17), 24, 4),
                                       ((23, 24), (8, 8), 40, 5), ((40, 40), (41, 40), 525, 2)])
def test_residual_norm_of_grown_bases(cr, kind, sy, sx, j, m):
    p = synth.rect2d(shape_y=sy, shape_x=sx, m=m)
    o = Oracle.from_problem(p)
    rng = np.random.default_rng(7)
    U, V = (columns(np.eye(L.n) if kind == "random" else eigvecs(L), j, kind) for L in (p.Ly, p.Lx))
    Z = rng.standard_normal((j, j)) / j
    want = np.linalg.norm(o.D() - o.A_op(U @ Z @ V.T)) / np.linalg.norm(o.D())
    with cr.ConReg.from_problem(p, r_cap=j) as g:
        for _ in range(2):  # the second time over the bases that the first left
            g.cr_set_factors(U, Z, V)
            got = g.cr_residual()["relres"]
            assert abs(got - want) <= 1e-10 * want, (got, want)
