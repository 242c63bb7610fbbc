"""The solution pass on both sides of its rule (600,000 entries with 36 M entries times columns), and
from there on around the edges of the digits' tiles (64 x 32), matrix steps (16 columns) and
level sums (112 columns), with zero rows and a reference.

Tolerance per entry, with u = 2^-53: P = U Z and W = P V^T as float64 sums of j products each
are within (2 j + 4) u (|U| |Z| |V|^T) of the exact W.  Sums of squares of n entries within
that bound agree to 2 sum |w| dw + sum dw^2 + 2 n u sum w^2."""
import numpy as np
import pytest

from paper_1808_05510_gb300 import synth

pytestmark = pytest.mark.gpu
U53 = 2.0 ** -53


@pytest.fixture(scope="module")
def cr():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1808_05510_gb300 import build, conreg

    build.build()
    conreg.load()
    return conreg


def factors(ny, nx, j, seed):
    rng = np.random.default_rng(seed)
    return rng.standard_normal((ny, j)), rng.standard_normal((j, j)), rng.standard_normal((nx, j))


def exact(U, Z, V):
    """float64 products with the rounding of a second float64 sum in the bound."""
    j = Z.shape[0]
    return U @ Z @ V.T, 2 * (2 * j + 4) * U53 * (np.abs(U) @ np.abs(Z) @ np.abs(V).T)


# ny x nx: 768 x 769 and 799 x 751 lie below and above 600,000 entries; 833 = 13 x 64 + 1
@pytest.mark.parametrize("sy,sx,j,jr", [((24, 32), (769, 1), 60, 0), ((47, 17), (751, 1), 60, 0), ((47, 17), (751, 1), 59, 0),
                                        ((49, 17), (27, 29), 55, 0), ((49, 17), (27, 29), 30, 26), ((32, 26), (25, 31), 112, 17),
                                        ((37, 23), (33, 25), 113, 128), ((65, 13), (21, 37), 129, 1), ((100, 16), (39, 41), 15, 8)])
def test_report_around_the_rule(cr, sy, sx, j, jr):
    p = synth.rect2d(shape_y=sy, shape_x=sx, m=2)
    U, Z, V = factors(p.ny, p.nx, j, 1)
    U[3] = 0.0
    V[5] = 0.0
    ref = factors(p.ny, p.nx, jr, 2) if jr else None
    with cr.ConReg.from_problem(p, r_cap=j) as g:
        g.cr_set_factors(U, Z, V)
        r = g.cr_solution_report(nonneg=True, ref=ref, want_w=True)
        r2 = g.cr_solution_report(nonneg=True, ref=ref)
    W, dw = exact(U, Z, V)
    P = np.maximum(W, 0)
    assert np.all(np.abs(r["W_out"] - P) <= dw)
    assert not r["W_out"][3].any() and not r["W_out"][:, 5].any()
    assert np.sum(W < -dw) <= r["n_negative"] <= np.sum(W < dw)
    Wr, dr = exact(*ref) if ref else (np.zeros_like(W), np.zeros_like(dw))
    for key, x, dx in (("w_fro2", W, dw), ("neg_fro2", np.minimum(W, 0), dw), ("ref_fro2", Wr, dr),
                       ("diff_fro2", P - Wr, dw + dr)):
        tot = np.sum(x * x)
        assert abs(r[key] - tot) <= 2 * np.sum(np.abs(x) * dx) + np.sum(dx * dx) + 4 * W.size * U53 * tot, key
    for key in ("n_negative", "w_min", "w_max", "diff_maxabs"):
        assert r[key] == r2[key]
