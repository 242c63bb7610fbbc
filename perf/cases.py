"""The work that is timed: calls of the public entry points over the range of problems the framework solves.

Every case is one pass of a user's program through ``ConReg``, ``solve_batch`` or ``ConvNet``: the problem handle
(Laplacians, X, Y, Omega, lambda on the GPU) is what such a program keeps, the call with its host vectors and factors
is what it repeats.  Sizes are those of ``synth``, the tests and ``bench.py``: the 20 x 20 toy, the 7,500-voxel
visual cortex (28 injections, lambda 100), the 15,000-voxel sweep data set (126 injections), the 45,000-voxel
whole-cortex shell (126 injections, lambda 1e3) and the shell of millions of voxels.  The geometry of a case (mask
and Laplacian) follows from its sizes, its injections, projections and factors from the seed.

Solver tolerances are tight (``tol``) so that an output is the solution of its system and not of a stopping test.

Kinds:
  greedy    Algorithm 1 from W = 0 to a small rank, factors and stopping quantities out
  solve     one ALS sub-system (Eqs. ALS_linsys, ALS_linsys_v) with the vectors of a first ALS sweep
  residual  the right sides R_j v and R_j^T u of an ALS sweep at rank j
  project   a checkpoint's factors restored, projected (Eq. Proj_Sylv) and checked (relres, J, dW)
  report    the pass over W = U Z V^T: projection onto W >= 0 and errors against another solution
  sweep     lambda x fold members solved side by side and scored on their held-out injections
  train     loss and gradients of the learned preconditioner's network, and its forward pass
"""
import functools
import math

import numpy as np
import torch

from paper_1808_05510_gb300 import conreg, synth

PREC = {"fp64": conreg.CR_FP64, "mixed": conreg.CR_MIXED}


def listed():
    return [
        # the toy's first ranks: every launch and read-back of a greedy step counts
        dict(name="greedy-toy-fp64", kind="greedy", shape="square", n=400, m=5, lam=100.0, rank=4, prec="fp64",
             tol=1e-12),
        # the headline workload: first ranks of the visual cortex in the mixed form
        dict(name="greedy-visual-mixed", kind="greedy", shape="blob", n=7500, m=28, lam=100.0, rank=6, prec="mixed",
             tol=1e-11),
        # the same problem in the float64 form (multigrid on both sides)
        dict(name="greedy-visual-fp64", kind="greedy", shape="blob", n=7500, m=28, lam=100.0, rank=3, prec="fp64",
             tol=1e-11),
        # the v-side system of the visual cortex, float64: multigrid with the Woodbury step
        dict(name="solve-v-visual-fp64", kind="solve", side="v", shape="blob", n=7500, m=28, lam=100.0, prec="fp64",
             tol=1e-11),
        # a sweep member's v-side system below lambda 1e3 in the mixed form: float32 Jacobi PCG on one cluster
        dict(name="solve-v-sweep-mixed", kind="solve", side="v", shape="blob", n=15000, m=100, lam=16.0, prec="mixed",
             tol=1e-12),
        # the whole-cortex shell's u-side system, mixed: multigrid with its tables outside shared memory
        dict(name="solve-u-cortex-mixed", kind="solve", side="u", shape="shell", n=45000, m=126, lam=1e3, prec="mixed",
             tol=1e-11),
        # the grid-wide PCG on vectors that stream from memory
        dict(name="solve-u-stress-mixed", kind="solve", side="u", shape="shell", n=3000000, m=4, lam=1e3, prec="mixed",
             tol=1e-11),
        # the right sides of one ALS sweep at the headline's rank cap: the smallest calls
        dict(name="residual-visual", kind="residual", shape="blob", n=7500, m=28, lam=100.0, rank=100, prec="fp64"),
        # a checkpoint at rank 240 of the time-to-relres run restored, projected and checked
        dict(name="project-visual-fp64", kind="project", shape="blob", n=7500, m=28, lam=100.0, rank=240, prec="fp64",
             tol=1e-12),
        # errors of the rank-100 solution, made nonnegative, against a rank-140 reference (the paper's E(W_r, W_140))
        dict(name="report-visual", kind="report", shape="blob", n=7500, m=28, lam=100.0, rank=100, ref=140, prec="fp64"),
        # two lambdas x three folds of the 15,000-voxel data set, problems created inside the call
        dict(name="sweep-mixed", kind="sweep", shape="blob", n=15000, m=126, lam=16.0, lam2=4000.0, folds=3, rank=4,
             prec="mixed", tol=1e-11),
        # a training step's loss and gradients on the 40^3 box, batches of 8
        dict(name="train-box40", kind="train", box=40, batch=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["greedy", "greedy", "residual", "residual", "project", "project", "report",
                                        "report", "sweep", "train"])
    if kind == "train":
        return dict(kind=kind, box=rng.randint(9, 40), batch=rng.randint(1, 8))
    lam = 10.0 ** rng.uniform(0.0, 3.5)
    prec = rng.choice(["fp64", "mixed"])
    if kind == "solve":
        shape = rng.choice(["blob", "blob", "shell", "stress"])
        n = _log(rng, 500, 30000) if shape == "blob" else _log(rng, 10000, 60000) if shape == "shell" else _log(
            rng, 150000, 1000000)
        if shape != "blob":
            lam = max(lam, 300.0)
        return dict(kind=kind, side=rng.choice(["u", "v"]), shape=shape.replace("stress", "shell"), n=n,
                    m=rng.randint(2, 6) if shape == "stress" else rng.randint(4, 126), lam=lam, prec=prec, tol=1e-12)
    if kind == "greedy":
        shape = rng.choice(["square", "rect", "blob"])
        n = _log(rng, 60, 2500) if shape != "blob" else _log(rng, 700, 9000)
        return dict(kind=kind, shape=shape, n=n, m=rng.randint(3, 30), lam=lam, rank=rng.randint(2, 5), prec=prec,
                    tol=1e-12)
    if kind == "residual":
        return dict(kind=kind, shape=rng.choice(["square", "blob", "shell"]), n=_log(rng, 300, 45000),
                    m=rng.randint(3, 126), lam=lam, rank=rng.randint(1, 160), prec=prec)
    if kind == "project":
        return dict(kind=kind, shape=rng.choice(["square", "blob"]), n=_log(rng, 700, 9000), m=rng.randint(3, 60),
                    lam=lam, rank=_log(rng, 8, 240), prec=prec, tol=1e-11)
    if kind == "report":
        return dict(kind=kind, shape=rng.choice(["square", "rect", "blob"]), n=_log(rng, 300, 9000),
                    m=rng.randint(3, 28), lam=lam, rank=rng.randint(1, 140), ref=rng.choice([0, rng.randint(1, 140)]),
                    prec=prec)
    return dict(kind=kind, shape="blob", n=_log(rng, 2000, 15000), m=rng.randint(20, 126), lam=lam,
                lam2=10.0 ** rng.uniform(0.0, 4.0), folds=rng.randint(2, 3), rank=rng.randint(1, 4), prec=prec,
                tol=1e-12)


# ---- geometry and data ----------------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=64)
def _geometry(shape, n, y_side=False):
    """(grid, Laplacian, voxel coordinates as float64) of a mask of about n voxels."""
    rng = np.random.default_rng(n)
    if shape == "square" or shape == "rect":
        side = max(6, int(round(math.sqrt(n))))
        mask = np.ones((side, side) if shape == "square" else (side + 2, side - 1) if y_side else (side - 2, side + 1),
                       dtype=bool)
    elif shape == "blob":
        box = max(10, int(round(40 * (n / 7500.0) ** (1.0 / 3.0))))
        mask = synth.blob_mask((box, box, box), n, rng, smooth=4.0 if box >= 30 else 2.0)
    elif n <= 100000:
        s = (n / 45000.0) ** (1.0 / 3.0)
        mask = synth.shell_mask(tuple(int(round(d * s)) for d in (96, 64, 80)), n)
    else:  # the stress workload's ellipsoidal shell, scaled
        side = int(round(256 * (n / 4e6) ** (1.0 / 3.0)))
        a = 0.46 * side
        t = 1.0 - (1.0 - min(0.999, n / (4.0 / 3.0 * math.pi * a ** 3))) ** (1.0 / 3.0)
        c = (side - 1) / 2.0
        z, y, x = np.ogrid[:side, :side, :side]
        rho2 = ((z - c) / a) ** 2 + ((y - c) / a) ** 2 + ((x - c) / a) ** 2
        mask = (rho2 <= 1.0) & (rho2 >= (1.0 - t) ** 2)
    g = synth.Grid(mask)
    return g, synth.grid_laplacian(g), torch.from_numpy(g.coords().astype(np.float64)).cuda()


def _unit(grid, coords):
    dims = torch.tensor([max(d - 1.0, 1.0) for d in grid.mask.shape], dtype=torch.float64, device=coords.device)
    return coords / dims


def _problem(case, seed):
    """The recipe of ``synth`` with the arithmetic on the GPU: truncated Gaussian injections, Omega = 1{X <= 0.4},
    Y = (W_true X + noise) o Omega."""
    rng = np.random.default_rng([seed, case["n"], case["m"]])
    gx, Lx, cx = _geometry(case["shape"], case["n"])
    gy, Ly, cy = _geometry(case["shape"], case["n"], True) if case["shape"] == "rect" else (gx, Lx, cx)
    m, nx, ny = case["m"], gx.n, gy.n
    wide = case["shape"] == "shell" and nx <= 100000
    X = torch.zeros(m, nx, dtype=torch.float64, device="cuda")
    for a in range(m):
        ctr, sig = cx[int(rng.integers(nx))], rng.uniform(2.0, 5.0) if wide else rng.uniform(1.8, 2.5)
        amp = rng.uniform(0.2, 1.0) if wide else 1.0
        d2 = ((cx - ctr) ** 2).sum(1)
        X[a] = torch.where(d2 <= 9.0 * sig * sig, amp * torch.exp(-d2 / (2.0 * sig * sig)), 0.0)
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 40)))
    if gx is gy:
        Om = X <= 0.4
    else:
        Om = torch.rand(m, ny, device="cuda", generator=gen) > 0.25
    if nx > 100000:  # as in the stress workload only the sub-solves run: Y is noise on Omega
        WX = torch.randn(m, ny, dtype=torch.float64, device="cuda", generator=gen)
    else:
        py, px = _unit(gy, cy), _unit(gx, cx)
        use = torch.nonzero((X != 0).any(0)).ravel()
        Xs, ps = X[:, use], px[use]
        WX = torch.empty(m, ny, dtype=torch.float64, device="cuda")
        for s in range(0, ny, 4096):
            q = py[s:s + 4096]
            WX[:, s:s + 4096] = Xs @ torch.exp(-torch.cdist(ps, q) ** 2 / 0.16)
        far = torch.exp(-((ps - 0.8) ** 2).sum(1) / 0.04)
        WX += 0.9 * (Xs @ far)[:, None] * torch.exp(-((py - 0.1) ** 2).sum(1) / 0.04)[None, :]
        WX += 0.01 * float((WX * Om).abs().max()) * torch.randn(m, ny, dtype=torch.float64, device="cuda",
                                                                generator=gen)
    Y = WX * Om
    host = lambda t, k: np.asfortranarray(t.to(k).cpu().numpy().T)  # noqa: E731
    return synth.Problem("", gx, gy, Lx, Ly, host(X, torch.float64), host(Y, torch.float64), host(Om, torch.uint8),
                         float(case["lam"]), int(case.get("rank", 4)))


def _smooth(grid, coords, seed):
    """Unit bump of a quarter of the box around a random voxel: the shape of a greedy solve's factors."""
    c = _unit(grid, coords)
    ctr = c[int(np.random.default_rng(seed).integers(grid.n))]
    v = torch.exp(-((c - ctr) ** 2).sum(1) / (2.0 * 0.25 ** 2))
    return (v / v.norm()).cpu().numpy()


def _vectors(case, p, seed):
    """(unit vector, right side) of the sub-system in a first ALS sweep: v = R_0^T 1, or a smooth u."""
    if case["side"] == "u":
        v = p.X @ p.Y.sum(axis=0)
        v /= np.linalg.norm(v)
        return v, p.Y @ (p.X.T @ v)
    u = _smooth(p.grid_y, _geometry(case["shape"], case["n"], case["shape"] == "rect")[2], seed + 1)
    return u, p.X @ (p.Y.T @ u)


def _basis(coords, grid, j, gen):
    """Orthonormal factors of slowly decaying smoothness: cosines of random wave vectors with a little noise."""
    c = _unit(grid, coords)
    k = torch.randn(c.shape[1], j, dtype=torch.float64, device="cuda", generator=gen) * (
        2.0 + 0.25 * torch.arange(j, dtype=torch.float64, device="cuda"))
    ph = 6.2831853 * torch.rand(j, dtype=torch.float64, device="cuda", generator=gen)
    B = torch.cos(c @ k + ph) + 0.05 * torch.randn(c.shape[0], j, dtype=torch.float64, device="cuda", generator=gen)
    return torch.linalg.qr(B)[0]


def _factors(case, seed, j, lead=1.0):
    gx, _, cx = _geometry(case["shape"], case["n"])
    gy, _, cy = _geometry(case["shape"], case["n"], True) if case["shape"] == "rect" else (gx, None, cx)
    j = min(j, gx.n, gy.n)
    gen = torch.Generator(device="cuda").manual_seed(1000003 * seed + j)
    U, V = _basis(cy, gy, j, gen), _basis(cx, gx, j, gen)
    decay = 0.95 ** torch.arange(j, dtype=torch.float64, device="cuda")
    Z = lead * torch.randn(j, j, dtype=torch.float64, device="cuda", generator=gen) * torch.minimum(
        decay[:, None], decay[None, :])
    return tuple(np.asfortranarray(t.cpu().numpy()) for t in (U, Z, V))


def _handle(case, p, r_cap, **kw):
    return conreg.ConReg.from_problem(p, r_cap=r_cap, precision=PREC[case["prec"]], precond=conreg.CR_PRECOND_AUTO,
                                      residual_every=0, **kw)


def _net_inputs(case, seed):
    b, B = case["box"], case["batch"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    c = torch.stack(torch.meshgrid(*[torch.linspace(-1.0, 1.0, b, device="cuda")] * 3, indexing="ij"))
    mask = (c ** 2).sum(0) <= 0.8
    x = torch.randn(B, 2, b, b, b, device="cuda", generator=gen) / math.sqrt(float(mask.sum()))
    x[:, 0] *= mask
    x[:, 1] = mask.float()
    t = torch.randn(B, b, b, b, device="cuda", generator=gen) * mask / math.sqrt(float(mask.sum()))
    w = 0.08 * np.random.default_rng(seed).standard_normal(conreg.ConvNet.param_count())
    return x, t, mask.to(torch.uint8), w.astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        x, t, mask, w = _net_inputs(case, seed)
        net = conreg.ConvNet((case["box"],) * 3, batch_cap=case["batch"], seed=seed)
        net.set_params(w)
        return dict(kind=kind, net=net, x=x, t=t, mask=mask)
    p = _problem(case, seed)
    if kind == "sweep":
        cols = np.random.default_rng(seed).permutation(case["m"])
        folds = [np.sort(f) for f in np.array_split(cols, case["folds"])]
        return dict(kind=kind, p=p, members=synth.sweep_members(case["m"], (case["lam"], case["lam2"]), folds),
                    rank=case["rank"], opts=dict(precision=PREC[case["prec"]], precond=conreg.CR_PRECOND_AUTO,
                                                 residual_every=0, r_cap=case["rank"], pcg_tol=case["tol"]),
                    tau=2.0 * case["tol"])
    if kind == "greedy":
        rank = min(case["rank"], p.nx, p.ny)
        return dict(kind=kind, g=_handle(case, p, rank, pcg_tol=case["tol"]), rank=rank, tau=2e-12,
                    zero=(np.zeros((p.ny, 0)), np.zeros((0, 0)), np.zeros((p.nx, 0))))
    if kind == "solve":
        w, rhs = _vectors(case, p, seed)
        return dict(kind=kind, side=case["side"], g=_handle(case, p, 2, pcg_tol=case["tol"]), w=w, rhs=rhs)
    F = _factors(case, seed, case["rank"])
    j = F[1].shape[0]
    g = _handle(case, p, j)
    if kind == "project":
        return dict(kind=kind, g=g, F=F, tol=case["tol"])
    g.cr_set_factors(*F)
    if kind == "report":
        return dict(kind=kind, g=g, ref=_factors(case, seed + 7, case["ref"], 0.9) if case["ref"] else None)
    rng = np.random.default_rng(seed + 3)
    v, u = rng.standard_normal(p.nx), rng.standard_normal(p.ny)
    return dict(kind=kind, g=g, v=v / np.linalg.norm(v), u=u / np.linalg.norm(u))


def run(state):
    kind = state["kind"]
    if kind == "train":
        loss, grads = state["net"].gradients(state["x"], state["t"], state["mask"])
        return {"loss": loss, "grads": grads, "out": state["net"].forward(state["x"])}
    if kind == "sweep":
        res, kept = conreg.solve_batch(state["p"], state["members"], r_max=state["rank"], tau=state["tau"], keep=True,
                                       **state["opts"])
        out = {"factors": [g.cr_get_factors() for g in kept],
               "scores": np.array([[r["cv_num"], r["cv_den"], r["J"], r["relres"]] for r in res])}
        for g in kept:
            g.close()
        return out
    g = state["g"]
    if kind == "solve":
        return (g.cr_solve_u if state["side"] == "u" else g.cr_solve_v)(state["w"], state["rhs"])[0]
    if kind == "residual":
        return [g.cr_apply_residual(state["v"]), g.cr_apply_residual(state["u"], trans=True)]
    if kind == "greedy":
        g.cr_set_factors(*state["zero"])
        info = g.cr_solve(state["rank"], state["tau"])
        return {"factors": g.cr_get_factors(), "info": np.array([info["relres"], info["J"]])}
    if kind == "project":
        g.cr_set_factors(*state["F"])
        g.cr_project(state["tol"])
        res = g.cr_residual()
        return {"factors": g.cr_get_factors(), "info": np.array([res["relres"], res["J"], res["dW"]])}
    r = g.cr_solution_report(nonneg=True, ref=state["ref"])
    return {"n_negative": r["n_negative"],
            "stats": np.array([r["w_min"], r["w_max"], r["w_fro2"], r["neg_fro2"], r["ref_fro2"], r["diff_fro2"],
                               r["diff_maxabs"], r["rms"], r["rel"] if state["ref"] is not None else 0.0])}


def work(case):
    """Bytes: each input and output of the call once (8 B a number; a stencil row's 24 B of neighbours).  Operations:
    the least that the path computes whatever its solver, one operator per system solved."""
    kind = case["kind"]
    if kind == "train":
        v = case["box"] ** 3 * case["batch"]
        return {"bytes": 4.0 * 4 * v + 2 * 64 * 1024, "flops": 2.0 * 27 * (2 * 16 + 16 * 16 * 2 + 16) * v * 4}
    n, m = float(case["n"]), float(case["m"])
    r = float(case.get("rank", 1))
    grid = 2 * n * (24 + 8)
    if kind == "solve":
        return {"bytes": n * (24 + 8 + 3 * 8 + m), "flops": 2.0 * n * (14 + m)}
    if kind == "residual":
        return {"bytes": 8.0 * n * (2 * r + 4) + n * m * 9, "flops": 2.0 * n * (4 * 3 * r + 4 * m)}
    if kind == "report":
        return {"bytes": 8.0 * 2 * n * (r + case["ref"]), "flops": 2.0 * n * n * (r + case["ref"])}
    if kind == "project":
        return {"bytes": grid + 8.0 * 2 * n * r + n * m * 9 + 16 * r * r,
                "flops": 2.0 * n * r * r * (m / 2 + 4) + 2.0 * r * r * (2 * r + 4 * m)}
    one = {"bytes": grid + 8.0 * 2 * n * r + n * m * 9,
           "flops": r * (2.0 * n * (28 + 2 * m) + 2.0 * n * r * (m + 8)) + 2.0 * r ** 3 * (2 * r + 4 * m)}
    k = 2 * case["folds"] if kind == "sweep" else 1
    return {"bytes": k * one["bytes"], "flops": k * one["flops"]}


# ---- the same results in 64 bits, in plain torch ----------------------------------------------------------------------

class _Dense:
    """The problem's operators in float64: Laplacians as neighbour tables, everything else dense."""

    def __init__(self, p):
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).double().cuda()  # noqa: E731
        self.X, self.Y, self.Om, self.lam = t(p.X), t(p.Y), t(p.Omega), p.lam
        self.Ly = self._table(p.Ly)
        self.Lx = self.Ly if p.Lx is p.Ly else self._table(p.Lx)
        self.nx, self.ny, self.m = p.nx, p.ny, p.m

    @staticmethod
    def _table(L):
        rp, col = np.asarray(L.rowptr, np.int64), np.asarray(L.col, np.int64)
        row = np.repeat(np.arange(L.n), np.diff(rp))
        off = col != row
        slot = np.arange(len(col)) - rp[row]
        nbr = np.full((L.n, int(np.diff(rp).max())), L.n, dtype=np.int64)
        nbr[row[off], slot[off]] = col[off]
        return torch.from_numpy((nbr < L.n).sum(1)).double().cuda(), torch.from_numpy(nbr).cuda()

    @staticmethod
    def lap(L, w):
        pad = torch.cat([w, torch.zeros_like(w[:1])])
        deg = L[0] if w.dim() == 1 else L[0][:, None]
        out = deg * w
        for k in range(L[1].shape[1]):
            out -= pad[L[1][:, k]]
        return out

    def dense(self, L):
        return self.lap(L, torch.eye(L[0].shape[0], dtype=torch.float64, device="cuda"))

    def coeffs(self, L, w):
        lw = self.lap(L, w)
        return float(w @ lw), float(lw @ lw)

    def sub(self, side, w):
        """(operator, diagonal, Laplacian, c, d, data diagonal or weights) of A_hat (u) or B_hat (v) for the vector w."""
        L, K = (self.Ly, self.Lx) if side == "u" else (self.Lx, self.Ly)
        c, d = self.coeffs(K, w)
        sq = L[0] ** 2 + L[0] + 2 * c * L[0] + d
        if side == "u":
            q = self.Om @ (self.X.T @ w) ** 2
            return lambda x: self.lam * (self.lap(L, self.lap(L, x) + 2 * c * x) + d * x) + q * x, self.lam * sq + q, L, c, d, q
        s = self.Om.T @ (w * w)
        return (lambda x: self.lam * (self.lap(L, self.lap(L, x) + 2 * c * x) + d * x) + self.X @ (s * (self.X.T @ x)),
                self.lam * sq + (self.X ** 2) @ s, L, c, d, s)

    def solve(self, side, w, b):
        """Conjugate gradients to the rounding floor, restarted from the true residual."""
        A, D, *_ = self.sub(side, w)
        x = torch.zeros_like(b)
        for _ in range(4):
            r = b - A(x)
            z = r / D
            p, rz, r0 = z, r @ z, float(r.norm())
            e = torch.zeros_like(b)
            for it in range(20000 if r0 > 0.0 else 0):
                q = A(p)
                a = rz / (p @ q)
                e += a * p
                r = r - a * q
                z = r / D
                rz2 = r @ z
                p = z + (rz2 / rz) * p
                rz = rz2
                if it % 16 == 15 and float(r.norm()) <= 1e-7 * r0:
                    break
            x = x + e
        return x

    def project(self, U, V, Z):
        """Z of Eq. (Proj_Sylv) by conjugate gradients preconditioned with the operator's diagonal in the eigenbases
        of U^T L_y U and V^T L_x V."""
        LU, LV = self.lap(self.Ly, U), self.lap(self.Lx, V)
        A1, A2, B1, B2 = U.T @ LU, LU.T @ LU, V.T @ LV, LV.T @ LV
        H, G = V.T @ self.X, torch.stack([U.T @ (self.Om[:, a, None] * U) for a in range(self.m)])
        F = (U.T @ (self.Om * self.Y)) @ H.T
        la, Qa = torch.linalg.eigh(A1)
        lb, Qb = torch.linalg.eigh(B1)
        dA, dB, Ht = (Qa.T @ A2 @ Qa).diagonal(), (Qb.T @ B2 @ Qb).diagonal(), Qb.T @ H
        g = torch.einsum("aii->a", G) / U.shape[1]
        D = self.lam * (dA[:, None] + 2 * la[:, None] * lb[None, :] + dB[None, :])
        Hg = Ht * g.sqrt()
        cap = torch.linalg.inv(torch.eye(self.m, dtype=torch.float64, device="cuda") + torch.einsum(
            "km,ik,kn->imn", Hg, 1.0 / D, Hg))

        def K(S):
            T = torch.einsum("aij,ja->ia", G, S @ H)
            return self.lam * (S @ B2 + 2 * A1 @ S @ B1 + A2 @ S) + T @ H.T

        def M(R):
            R = (Qa.T @ R @ Qb) / D
            R = R - (torch.einsum("imn,in->im", cap, R @ Hg) @ Hg.T) / D
            return Qa @ R @ Qb.T

        for _ in range(3):
            R = F - K(Z)
            r0, W = float(R.norm()), M(R)
            P, rz, E = W, (R * W).sum(), torch.zeros_like(Z)
            for _ in range(400 if r0 > 0.0 else 0):
                Q = K(P)
                a = rz / (P * Q).sum()
                E += a * P
                R = R - a * Q
                W = M(R)
                rz2 = (R * W).sum()
                P = W + (rz2 / rz) * P
                rz = rz2
                if float(R.norm()) <= 1e-8 * r0:
                    break
            Z = Z + E
        return Z

    def op(self, U, Z, V, v):
        """A(U Z V^T) v."""
        W = lambda w: U @ (Z @ (V.T @ w))  # noqa: E731
        lv = self.lap(self.Lx, v)
        out = self.lam * (W(self.lap(self.Lx, lv)) + self.lap(self.Ly, 2 * W(lv) + self.lap(self.Ly, W(v))))
        return out + (self.Om * (U @ (Z @ (V.T @ self.X)))) @ (self.X.T @ v)

    def R(self, U, Z, V, v):
        return (self.Om * self.Y) @ (self.X.T @ v) - self.op(U, Z, V, v)

    def Rt(self, U, Z, V, u):
        W = lambda w: V @ (Z.T @ (U.T @ w))  # noqa: E731
        lu = self.lap(self.Ly, u)
        out = self.lam * (self.lap(self.Lx, self.lap(self.Lx, W(u)) + 2 * W(lu)) + W(self.lap(self.Ly, lu)))
        E = self.Om * (self.Y - U @ (Z @ (V.T @ self.X)))
        return self.X @ (E.T @ u) - out

    def info(self, U, Z, V):
        """(relres, J): ||D - A(W)||_F / ||D||_F over blocks of columns, and the objective."""
        num = den = S2 = 0.0
        D = self.Om * self.Y
        E = D - self.Om * (U @ (Z @ (V.T @ self.X)))
        LU = self.lap(self.Ly, U)
        L2U, LV = self.lap(self.Ly, LU), self.lap(self.Lx, V)
        L2V = self.lap(self.Lx, LV)
        for s in range(0, self.nx, 2048):
            k = slice(s, s + 2048)
            B = U @ (Z @ L2V[k].T) + 2 * (LU @ (Z @ LV[k].T)) + L2U @ (Z @ V[k].T)
            num += float(((E @ self.X[k].T - self.lam * B) ** 2).sum())
            den += float(((D @ self.X[k].T) ** 2).sum())
            S2 += float(((LU @ (Z @ V[k].T) + U @ (Z @ LV[k].T)) ** 2).sum())
        return math.sqrt(num / den), 0.5 * float((E * E).sum()) + 0.5 * self.lam * S2

    def greedy(self, rank):
        """Algorithm 1 with direct sub-solves (dense Cholesky)."""
        eye = lambda L: torch.eye(L[0].shape[0], dtype=torch.float64, device="cuda")  # noqa: E731
        dl = {}
        for side, L in (("u", self.Ly), ("v", self.Lx)):
            if side == "v" and self.Lx is self.Ly:
                dl["v"] = dl["u"]
            else:
                M = self.dense(L)
                dl[side] = (M, self.lap(L, M), eye(L))

        def direct(side, w, b):
            _, _, _, c, d, q = self.sub(side, w)
            M, M2, I = dl[side]
            A = self.lam * (M2 + 2 * c * M + d * I)
            A = A + torch.diag(q) if side == "u" else A + (self.X * q) @ self.X.T
            C = torch.linalg.cholesky(A)
            x = torch.cholesky_solve(b[:, None], C)
            return (x + torch.cholesky_solve(b[:, None] - A @ x, C))[:, 0]

        def orth(Q, u):
            for _ in range(2):
                u = u - Q @ (Q.T @ u)
            return torch.cat([Q, (u / u.norm())[:, None]], 1)

        z = lambda n, k: torch.zeros(n, k, dtype=torch.float64, device="cuda")  # noqa: E731
        U, Z, V = z(self.ny, 0), z(0, 0), z(self.nx, 0)
        for j in range(rank):
            v = self.Rt(U, Z, V, torch.ones(self.ny, dtype=torch.float64, device="cuda"))
            v = v / v.norm()
            for _ in range(10):
                uh = direct("u", v, self.R(U, Z, V, v))
                u = uh / uh.norm()
                vh = direct("v", u, self.Rt(U, Z, V, u))
                v = vh / vh.norm()
                if abs(float(uh.norm() / vh.norm()) - 1.0) <= 0.1:
                    break
            U, V = orth(U, u), orth(V, v)
            Z0 = z(j + 1, j + 1)
            Z0[:j, :j] = Z
            Z = self.project(U, V, Z0)
        return U, Z, V


def _net_exact(x, t, mask, w):
    """Loss, gradients and output of the network in float64: 27 shifted products a layer."""
    ch = [2, 16, 16, 16, 1]
    w = torch.from_numpy(w).double().cuda().requires_grad_()
    a, k = x.double(), 0
    for l in range(4):
        co, ci = ch[l + 1], ch[l]
        W, bias = w[k:k + co * ci * 27].reshape(co, ci, 27), w[k + co * ci * 27:k + co * ci * 27 + co]
        k += co * ci * 27 + co
        pad = torch.nn.functional.pad(a, (1,) * 6)
        D, H, Q = a.shape[2:]
        z = bias.reshape(1, co, 1, 1, 1)
        for s in range(27):
            dz, dy, dx = s // 9, s // 3 % 3, s % 3
            z = z + torch.einsum("oc,bczyx->bozyx", W[:, :, s], pad[:, :, dz:dz + D, dy:dy + H, dx:dx + Q])
        a = torch.relu(z) if l < 3 else z
    a = a[:, 0]
    m, t = mask.double(), t.double()
    loss = (m * (a - t) ** 2).sum() / (m * t * t).sum()
    loss.backward()
    return {"loss": loss.detach(), "grads": w.grad, "out": a.detach()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _net_exact(*_net_inputs(case, seed))
    if kind == "sweep" or (kind == "greedy" and case["n"] > 9500):
        return None  # tens of dense factorisations of 15,000 rows: minutes
    p = _problem(case, seed)
    o = _Dense(p)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    if kind == "solve":
        w, rhs = _vectors(case, p, seed)
        return o.solve(case["side"], t(w), t(rhs))
    if kind == "greedy":
        F = o.greedy(min(case["rank"], p.nx, p.ny))
        return {"factors": F, "info": torch.tensor(o.info(*F), dtype=torch.float64)}
    U, Z, V = (t(a) for a in _factors(case, seed, case["rank"]))
    if kind == "residual":
        rng = np.random.default_rng(seed + 3)
        v, u = rng.standard_normal(p.nx), rng.standard_normal(p.ny)
        return [o.R(U, Z, V, t(v / np.linalg.norm(v))), o.Rt(U, Z, V, t(u / np.linalg.norm(u)))]
    if kind == "project":
        Z1 = o.project(U, V, Z)
        res = o.info(U, Z1, V) + (float((Z1 - Z).norm() / Z1.norm()),)
        return {"factors": (U, Z1, V), "info": torch.tensor(res, dtype=torch.float64)}
    W = U @ Z @ V.T
    ref = torch.zeros_like(W)
    if case["ref"]:
        a, b, c = (t(a) for a in _factors(case, seed + 7, case["ref"], 0.9))
        ref = a @ b @ c.T
    P = W.clamp(min=0.0)
    diff = float(((P - ref) ** 2).sum())
    return {"n_negative": None, "stats": torch.tensor(
        [float(W.min()), float(W.max()), float((W * W).sum()), float(((W - P) ** 2).sum()), float((ref * ref).sum()),
         diff, float((P - ref).abs().max()), math.sqrt(diff / W.numel()),
         math.sqrt(diff / float((ref * ref).sum())) if case["ref"] else 0.0], dtype=torch.float64)}
