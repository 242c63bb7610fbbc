"""cr_solution_report where the device has no room for the digits of the factors
(cr_post_tc.cu): the call is answered by the float64 pass, as it is for small ranks.

Tolerance, u = 2^-53: entries within (2 j + 4) u (|U| |Z| |V|^T) of the exact W in both passes,
so |W|^2 of n entries agrees to 4 sum |w| dw + 4 n u sum w^2."""
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


@pytest.mark.parametrize("jr", [0, 40])
def test_report_without_room_for_digits(cr, monkeypatch, jr):
    p = synth.masked3d(box=14, n_target=1200)  # enough entries for the digits
    rng = np.random.default_rng(1)
    j = 30
    U, Z, V = rng.standard_normal((p.ny, j)), rng.standard_normal((j, j)), rng.standard_normal((p.nx, j))
    ref = (rng.standard_normal((p.ny, jr)), rng.standard_normal((jr, jr)), rng.standard_normal((p.nx, jr))) if jr else None
    limit, refused = [None], []
    base = cr._TorchAllocator._do_alloc

    def alloc(self, nbytes, ctx):
        if limit[0] and int(nbytes) > limit[0]:
            refused.append(int(nbytes))
            return None
        return base(self, nbytes, ctx)

    monkeypatch.setattr(cr._TorchAllocator, "_do_alloc", alloc)
    got = []
    for small in (False, True):
        with cr.ConReg.from_problem(p, r_cap=j) as g:
            g.cr_set_factors(U, Z, V)
            limit[0] = 12 * p.ny * max(j, jr) if small else None  # U Z takes 8 bytes an entry, the digits 16
            got.append([g.cr_solution_report(nonneg=True, ref=ref) for _ in range(2)])
            limit[0] = None
    assert refused
    W = U @ Z @ V.T
    dw = (2 * j + 4) * U53 * (np.abs(U) @ np.abs(Z) @ np.abs(V).T)
    tol = 4 * np.sum(np.abs(W) * dw) + 4 * W.size * U53 * np.sum(W * W)
    for q in got[0] + got[1]:
        assert abs(q["w_fro2"] - got[0][0]["w_fro2"]) <= tol
        assert np.sum(W < -2 * dw) <= q["n_negative"] <= np.sum(W < 2 * dw)
    a, b = ({k: v for k, v in q.items() if v == v} for q in got[1])
    assert a == b  # a second call is refused its digits again, with the same answer
