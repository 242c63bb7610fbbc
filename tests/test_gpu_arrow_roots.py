"""The secular roots of the arrowhead step (csrc/cr_arrow.cu): one, two and three
poles, a warp's edge, couplings down to the deflation limit, poles over six
decades, roots that lie against a pole, alpha far outside the poles.

Tolerance: eigenvalues and M W = W mu to 1e-13 n of the largest entry, W^T W = I to
1e-13 n.  A root is an offset from its nearest pole and is taken when a step moves
that by four units of rounding or the function is down to its own rounding, so that
the coupling made from the roots is the given one to some n units."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1808_05510_gb300 import build

    build.build()
    from paper_1808_05510_gb300 import conreg

    conreg.load()
    return conreg


@pytest.mark.parametrize("kind", ["plain", "weak", "wide", "tiny", "close", "outside"])
@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 65, 240])
def test_roots(lib, n, kind):
    rng = np.random.default_rng(7 * n)
    d, z, alpha = np.sort(12.0 * rng.random(n)), rng.standard_normal(n), 5.0
    if kind == "weak":
        z *= 10.0 ** rng.uniform(-12.0, 0.0, n)
    elif kind == "wide":
        d = np.sort(10.0 ** rng.uniform(-5.0, 1.0, n))
    elif kind == "tiny":
        z *= 1e-7
    elif kind == "close":
        d = 3.0 + 1e-6 * np.arange(n)
    elif kind == "outside":
        alpha = -1e4
    M = np.diag(np.append(d, alpha))
    M[:n, n] = M[n, :n] = z
    mu, W = lib.arrow_check(d, z, alpha)
    scale = np.abs(M).max()
    assert np.all(np.diff(mu) >= -1e-14 * scale)
    assert np.abs(mu - np.linalg.eigvalsh(M)).max() <= 1e-13 * n * scale
    assert np.abs(W.T @ W - np.eye(n + 1)).max() <= 1e-13 * n
    assert np.abs(M @ W - W * mu).max() <= 1e-13 * n * scale
