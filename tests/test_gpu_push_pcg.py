"""The float32 cluster PCG that pushes values between CTAs (cr_pcg_push.cu), inside
the mixed form's float64 refinement, where its tables can go wrong: one CTA, more
CTAs than the last chunk fills, rows of one CTA needed by every other (a graph
without locality), columns of X without a row in some CTA, a single injection,
rows of X with many entries, several rows per thread.

Tolerance: the refinement solves to a float64 relative residual of 1e-13 and the
reference is a dense float64 solve, so the solutions agree to 20 cond 1.1e-13, at
least 1e-9 (as for the other PCG kernels)."""
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


def cubic_graph(n, seed):
    """Laplacian of three random perfect matchings on n rows: neighbours anywhere, degree at most 3."""
    rng = np.random.default_rng(seed)
    A = np.zeros((n, n))
    for _ in range(3):
        q = rng.permutation(n)
        A[q[0::2], q[1::2]] = A[q[1::2], q[0::2]] = 1.0
    L = np.diag(A.sum(1)) - A
    r, c = np.nonzero(L)
    return synth.CSR(n, np.searchsorted(r, np.arange(n + 1)).astype(np.int32), c.astype(np.int32), L[r, c])


def problem(name):
    if name == "one-injection":
        return synth.toy2d(side=11, m=1), 0
    if name == "chain":
        return synth.paper_toy(n=203, m=4), 5
    if name == "random-graph":
        p = synth.toy2d(side=30, m=7)
        L = cubic_graph(900, 3)
        return dataclasses.replace(p, Lx=L, Ly=L), 16
    if name == "dense-x":  # every row of X full, two rows per thread on one CTA
        p = synth.toy2d(side=29, m=45)
        X = np.random.default_rng(4).random(p.X.shape)
        return dataclasses.replace(p, X=X), 1
    return synth.masked3d(box=14, n_target=1200, m=9), 16  # blobs that reach a few CTAs each


@pytest.mark.parametrize("name", ["one-injection", "chain", "random-graph", "dense-x", "blobs"])
def test_pushing_pcg_matches_dense_solve(cr, name):
    p, cs = problem(name)
    o = Oracle.from_problem(p)
    rng = np.random.default_rng(8)
    v, u = synth.random_unit(p.nx, 5), synth.random_unit(p.ny, 6)
    bu, bv = rng.standard_normal(p.ny), rng.standard_normal(p.nx)
    with cr.ConReg.from_problem(p, r_cap=2, pcg_tol=1e-13, pcg_maxit=200000, precision=cr.CR_MIXED,
                                precond=cr.CR_PRECOND_JACOBI, cluster_size=cs) as g:
        first = g.cr_solve_u(v, bu)[0], g.cr_solve_v(u, bv)[0]
        again = g.cr_solve_u(v, bu)[0], g.cr_solve_v(u, bv)[0]
        zero = g.cr_solve_u(v, 0.0 * bu)[0]
        st = g.cr_get_stats()
    assert min(st["pcg_cluster"]) >= 1 and (cs == 0 or st["pcg_cluster"] == [cs, cs]), st
    Bs, s = o.B_hat(u)
    for x, y, A, b in ((first[0], again[0], o.A_hat(v).toarray(), bu),
                       (first[1], again[1], Bs.toarray() + (p.X * s) @ p.X.T, bv)):
        ref = np.linalg.solve(A, b)
        bar = max(1e-9, 20.0 * np.linalg.cond(A) * 1.1e-13)
        assert np.linalg.norm(x - ref) <= bar * np.linalg.norm(ref)
        assert np.array_equal(x, y)  # fixed summation order
    assert not zero.any()
