"""A Laplacian is refused when its entry list (stored zeros left out, equal indices
kept apart, columns in any order) differs from its transpose's."""
import ctypes as C

import numpy as np
import pytest

from paper_1808_05510_gb300 import build, conreg, synth


@pytest.fixture(scope="module")
def lib():
    build.build()
    return conreg.load()


def csr(n, entries, rng=None):
    """Rows in order; the entries of a row in a random order if rng is given."""
    rows = [[(j, v) for i, j, v in entries if i == r] for r in range(n)]
    if rng is not None:
        for row in rows:
            rng.shuffle(row)
    rp = np.cumsum([0] + [len(row) for row in rows]).astype(np.int32)
    flat = [e for row in rows for e in row]
    return synth.CSR(n, rp, np.array([int(j) for j, _ in flat], np.int32), np.array([float(v) for _, v in flat]))


def refused(lib, Lx, Ly):
    n = Lx.n
    X = Y = np.ones((n, 1))
    Om = np.ones((n, 1), np.uint8)
    d = conreg.cr_problem_desc()
    d.nx = d.ny = n
    d.ninj = 1
    for name, L in (("Lx", Lx), ("Ly", Ly)):
        setattr(d, name, conreg.cr_csr(n, conreg._ptr(L.rowptr, conreg._ip), conreg._ptr(L.col, conreg._ip),
                                       conreg._ptr(L.val)))
    d.X_host, d.ldx = conreg._ptr(X), n
    d.Y_host, d.ldy = conreg._ptr(Y), n
    d.Omega_host, d.ldo = conreg._ptr(Om, conreg._up), n
    d.lambda_ = 1.0
    opts, h = conreg.default_options(r_cap=1), C.c_void_p()
    st = lib.cr_create(C.byref(d), C.byref(opts), C.byref(h))
    lib.cr_destroy(h)  # without a GPU an accepted matrix fails later, with another message
    return st != conreg.CR_OK and b"not symmetric" in lib.cr_last_error(None)


@pytest.mark.parametrize("seed", range(4))
@pytest.mark.parametrize("n", [1, 2, 7, 30])
def test_symmetry(lib, n, seed):
    rng = np.random.default_rng(100 * n + seed)
    eye = csr(n, [(i, i, 1.0) for i in range(n)])

    def check(entries, want):
        L = csr(n, entries, rng)
        assert [refused(lib, L, eye), refused(lib, eye, L), refused(lib, L, L)] == [want] * 3

    ent = [(i, i, float(rng.integers(1, 4))) for i in range(n)]
    used = np.zeros(n, int)
    for _ in range(2 * n):  # repeated indices included
        i, j, v = int(rng.integers(n)), int(rng.integers(n)), float(rng.integers(1, 3))
        if max(used[i], used[j]) < 8:
            used[i] += 1
            used[j] += 1
            ent += [(i, j, v)] if i == j else [(i, j, v), (j, i, v)]
    check(ent, False)
    check(ent + [(0, n - 1, 0.0)], False)  # a stored zero without a partner
    if n > 1:
        check(ent + [(0, n - 1, 1.0)], True)
        check(ent + [(0, 1, 1.0), (1, 0, np.nextafter(1.0, 2.0))], True)
    if n > 2:  # as many entries in every row and column, at other places
        check(ent + [(i, (i + 1) % n, 9.0) for i in range(n)], True)
