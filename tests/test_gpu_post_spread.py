"""The solution pass (cr_post.cu, cr_post_tc.cu) where the entries of a factor's row differ
by many orders of magnitude: columns that decay, bumps whose large rows do not
meet, and nonnegative factors, whose W has no negative entry whatever its size.

Tolerance per entry, with u = 2^-53: P = U Z and W = P V^T as float64 sums of j
products each are within (2 j + 4) u (|U| |Z| |V|^T) of the exact W, entry by entry."""
import numpy as np
import pytest

from paper_1808_05510_gb300 import synth

pytestmark = pytest.mark.gpu
U53 = 2.0 ** -53
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


def bumps(n, j, width):
    return np.exp(-0.5 * ((np.linspace(0, 1, n)[:, None] - np.linspace(0, 1, j)[None]) / width) ** 2)


def factors(kind, ny, nx, j):
    rng = np.random.default_rng(j)
    if kind.startswith("bumps"):  # nonnegative, rows spread over 1 .. exp(-0.5 / width^2)
        w = float(kind[5:])
        return bumps(ny, j, w), np.diag(rng.uniform(0.5, 2.0, j)), bumps(nx, j, w)
    U, V = rng.standard_normal((ny, j)), rng.standard_normal((nx, j))
    if kind == "decay":  # the same in every row; V grows as U decays, but for a few rows
        d = 10.0 ** -np.linspace(0, 24, j)
        V[: nx // 2] = V[: nx // 2] * d
        V[nx // 2:] = V[nx // 2:] / d
        return U * d, np.diag(rng.uniform(0.5, 2.0, j)), V
    # "apart": U's large column meets V's zero one, what is left is 1e-21 of the rows' largest entries
    U[:, 1:] *= 1e-21
    V[:, 0] = 0.0
    V[: nx // 3, 0] = 1.0  # and rows where they do meet
    return U, np.eye(j), V


@pytest.mark.parametrize("kind", ["bumps0.1", "bumps0.08", "bumps0.05", "bumps0.02", "decay", "apart"])
@pytest.mark.parametrize("sides,j", [((13, 15, 14, 11), 24), ((20, 16, 9, 15), 115), ((27, 31, 25, 32), 60)])
def test_entries_to_their_own_size(cr, kind, sides, j):
    p = synth.rect2d(shape_y=sides[:2], shape_x=sides[2:], m=3)
    U, Z, V = factors(kind, p.ny, p.nx, j)
    ref = factors("bumps0.08" if kind != "bumps0.08" else "decay", p.ny, p.nx, 30)
    with cr.ConReg.from_problem(p, r_cap=j) as g:
        g.cr_set_factors(U, Z, V)
        r = g.cr_solution_report(want_w=True)
        r2 = g.cr_solution_report(nonneg=True, ref=ref)

    def exact(U, Z, V):
        a = [x.astype(LD) for x in (U, Z, V)]
        return a[0] @ a[1] @ a[2].T, (2 * Z.shape[0] + 4) * U53 * (np.abs(a[0]) @ np.abs(a[1]) @ np.abs(a[2]).T)

    W, dw = exact(U, Z, V)
    Wr, dr = exact(*ref)
    assert np.all(np.abs(r["W_out"] - W) <= dw)
    for q in (r, r2):
        assert np.sum(W < -dw) <= q["n_negative"] <= np.sum(W < dw)
        assert abs(q["w_min"] - W.min()) <= dw[np.abs(W - W.min()) <= 2 * dw].max()
    if kind.startswith("bumps"):
        assert r["n_negative"] == 0 and r["w_min"] > 0.0
    assert abs(r2["diff_maxabs"] - np.abs(np.maximum(W, 0) - Wr).max()) <= (dw + dr).max() * (1 + U53)
