"""A caller's allocator whose blocks start anywhere (here 8 bytes past a multiple of 256): the
library aligns what it uses, since its 16-byte loads and copies need it, and gives back
exactly the blocks that it got.  Results are bit for bit those with aligned blocks."""
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


def passes(cr, prec, precond, kernel):
    p = synth.masked3d(box=14, n_target=1200)  # enough entries for the solution pass's digits
    rng = np.random.default_rng(1)
    u, v = synth.random_unit(p.ny, 3), synth.random_unit(p.nx, 4)
    out = []
    with cr.ConReg.from_problem(p, r_cap=30, pcg_tol=1e-12, precision=getattr(cr, prec), precond=getattr(cr, precond),
                                pcg_kernel=kernel) as g:
        out += [g.cr_solve_u(v, rng.standard_normal(p.ny))[0], g.cr_solve_v(u, rng.standard_normal(p.nx))[0]]
        g.cr_set_factors(rng.standard_normal((p.ny, 30)), rng.standard_normal((30, 30)), rng.standard_normal((p.nx, 30)))
        r = g.cr_solution_report(want_w=True)
        out += [r["W_out"], np.array([r["w_fro2"], r["w_min"]])]
        if prec == "CR_MIXED":
            out.append(g.cr_galerkin_assembly(0))
    return [np.asarray(x) for x in out]


@pytest.mark.parametrize("prec", ["CR_FP64", "CR_MIXED"])
@pytest.mark.parametrize("precond,kernel", [("CR_PRECOND_JACOBI", 0), ("CR_PRECOND_JACOBI", 2), ("CR_PRECOND_MULTIGRID", 0)])
def test_blocks_that_start_anywhere(cr, monkeypatch, prec, precond, kernel):
    want = passes(cr, prec, precond, kernel)
    held, returned = {}, []
    base_alloc, base_free = cr._TorchAllocator._do_alloc, cr._TorchAllocator._do_free

    def alloc(self, nbytes, ctx):
        q = base_alloc(self, int(nbytes) + 8, ctx)
        if not q:
            return q
        held[int(q) + 8] = int(nbytes)
        return int(q) + 8

    def free(self, ptr, nbytes, ctx):
        returned.append(held.pop(int(ptr)) == int(nbytes))
        return base_free(self, int(ptr) - 8, nbytes, ctx)

    monkeypatch.setattr(cr._TorchAllocator, "_do_alloc", alloc)
    monkeypatch.setattr(cr._TorchAllocator, "_do_free", free)
    got = passes(cr, prec, precond, kernel)
    assert returned and all(returned) and not held
    for a, b in zip(want, got):
        assert np.array_equal(a, b)
