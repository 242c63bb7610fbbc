"""The solution pass on exact 8-bit digits (cr_post_tc.cu): every entry of W and the
statistics around the edges of its tiles (64 x 32), of its matrix steps (16
columns) and of its level sums (112 columns), with rows of very different size, zero
rows, a reference, and factors that it hands to the float64 pass.

Tolerance per entry, with u = 2^-53: P = U Z and W = P V^T as float64 sums of j
products each are within (2 j + 4) u (|U| |Z| |V|^T) of the exact W; the dropped
digits add at most 7 j 2^-64 of the largest entries' product of the two rows.
Sums of squares of n entries, formed in any order from entries within that
bound, agree to 2 sum |w| dw + 2 n u sum w^2."""
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


def factors(ny, nx, j, seed, spread=0.0):
    rng = np.random.default_rng(seed)
    U = rng.standard_normal((ny, j)) * 10.0 ** (spread * rng.uniform(-1, 1, (ny, 1)))
    V = rng.standard_normal((nx, j)) * 10.0 ** (spread * rng.uniform(-1, 1, (nx, 1)))
    return U, rng.standard_normal((j, j)), V


def exact(U, Z, V):
    W = (U.astype(np.longdouble) @ Z.astype(np.longdouble)) @ V.T.astype(np.longdouble)
    j = Z.shape[0]
    big = np.abs(U) @ np.abs(Z)
    bound = (2 * j + 4) * U53 * (big @ np.abs(V).T) + 7 * j * 2.0 ** -64 * np.outer(big.max(1), np.abs(V).max(1))
    return W, bound


@pytest.mark.parametrize("shape,j,jr,spread", [((8, 8, 8, 8), 24, 0, 0.0), ((9, 7, 6, 11), 25, 17, 0.0),
                                               ((12, 11, 11, 12), 112, 0, 0.0), ((12, 11, 11, 12), 113, 30, 0.0),
                                               ((13, 10, 12, 11), 60, 128, 5.0), ((5, 13, 16, 4), 32, 32, 40.0)])
def test_entries_and_statistics(cr, shape, j, jr, spread):
    p = synth.rect2d(shape_y=shape[:2], shape_x=shape[2:], m=3)
    j, jr = min(j, p.nx, p.ny), min(jr, p.nx, p.ny)
    U, Z, V = factors(p.ny, p.nx, j, 1, spread)
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
    # entries whose sign the bound leaves open may count either way
    assert np.sum(W < -dw) <= r["n_negative"] <= np.sum(W < dw)
    assert abs(r["w_min"] - W.min()) <= dw.max() and abs(r["w_max"] - W.max()) <= dw.max()
    Wr, dr = exact(*ref) if ref else (np.zeros_like(W), np.zeros_like(dw))
    n = W.size
    for key, x, dx in (("w_fro2", W, dw), ("neg_fro2", np.minimum(W, 0), dw), ("ref_fro2", Wr, dr),
                       ("diff_fro2", P - Wr, dw + dr)):
        tot = np.sum(x * x)
        assert abs(r[key] - tot) <= 2 * np.sum(np.abs(x) * dx) + np.sum(dx * dx) + 2 * n * U53 * tot, key
    for key in ("n_negative", "w_min", "w_max", "diff_maxabs"):
        assert r[key] == r2[key]
    for key in ("w_fro2", "neg_fro2", "ref_fro2", "diff_fro2"):
        assert abs(r[key] - r2[key]) <= 2 * n * U53 * abs(r[key])


def test_factors_beyond_the_digits_take_the_float64_pass(cr):
    p = synth.toy2d(side=9, m=2)
    U, Z, V = factors(p.ny, p.nx, 30, 3)
    U[4] *= 1e150
    V[7] *= 1e-150
    with cr.ConReg.from_problem(p, r_cap=30) as g:
        g.cr_set_factors(U, Z, V)
        r = g.cr_solution_report(want_w=True)
        W, dw = exact(U, Z, V)
        assert np.all(np.abs(r["W_out"] - W) <= dw)
        assert r["n_negative"] == np.sum(r["W_out"] < 0) and r["w_max"] == r["W_out"].max()
        U[2, 3] = np.inf
        g.cr_set_factors(U, Z, V)
        r = g.cr_solution_report(want_w=True)
        assert not np.isfinite(r["W_out"][2]).all() and np.isfinite(r["W_out"][3]).all()
