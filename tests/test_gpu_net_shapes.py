"""The network's weight gradients (cr_net.cu) over the shapes that decide their split: more
rows (sample, z, y) than CTAs and fewer, rows on both sides of a tile's width (32 columns in
float64, 64 in float32), a single column, and rows with a value that is not finite where
the gradient is zero.

Tolerances are those of test_gpu_learned.py: the float64 instantiation to 1e-10, the BF16
network to 1e-2 of the oracle with BF16 storage."""
import numpy as np
import pytest

from test_gpu_learned import bf16, env, oracle_all, random_case, unpack  # noqa: F401

pytestmark = pytest.mark.gpu


def close(g, dWs, dbs, tol):
    gW, gb = unpack(g)
    for l in range(4):
        assert np.linalg.norm(gW[l] - dWs[l]) <= tol * np.linalg.norm(dWs[l]), l
        assert np.linalg.norm(gb[l] - dbs[l]) <= tol * np.linalg.norm(dbs[l]) + 1e-7 * (tol > 1e-9), l


@pytest.mark.parametrize("dims,B", [((9, 13, 3), 3), ((2, 3, 31), 1), ((2, 3, 32), 2), ((3, 2, 33), 2), ((2, 2, 65), 2),
                                    ((3, 5, 1), 2)])
def test_float64_gradients(env, dims, B):  # noqa: F811
    torch, cr = env
    flat, x, t, mask = random_case(cr, sum(dims), dims, B)
    out, loss, g = cr.ConvNet.check_f64(dims, flat, x, t, mask)
    Ws, bs = unpack(flat)
    ref, loss_ref, dWs, dbs = oracle_all(x, Ws, bs, t, mask)
    assert np.linalg.norm(out - ref) <= 1e-10 * np.linalg.norm(ref)
    close(g, dWs, dbs, 1e-10)


@pytest.mark.parametrize("dims,B", [((9, 13, 3), 3), ((2, 3, 41), 2), ((2, 2, 64), 1), ((2, 2, 65), 2), ((1, 2, 130), 1)])
def test_bf16_gradients(env, dims, B):  # noqa: F811
    torch, cr = env
    flat, x, t, mask = (a.astype(np.float32) if a.dtype == np.float64 else a for a in random_case(cr, sum(dims), dims, B))
    net = cr.ConvNet(dims, batch_cap=B, seed=3)
    net.set_params(flat)
    loss, g = net.gradients(*(torch.tensor(a, device="cuda") for a in (x, t, mask)))
    net.close()
    Ws, bs = unpack(flat)
    _, _, dWs, dbs = oracle_all(x.astype(np.float64), [bf16(w, torch) for w in Ws], bs, t.astype(np.float64), mask,
                                round_fn=lambda a: bf16(a, torch))
    close(g, dWs, dbs, 1e-2)


@pytest.mark.parametrize("dims", [(7, 9, 1), (70, 2, 1), (11, 1, 1), (67, 1, 1), (1, 6, 1), (1, 1, 5), (1, 1, 1), (4, 1, 6), (5, 9, 2),
                                  (9, 5, 2), (3, 8, 7), (2, 7, 7), (6, 6, 7)])
def test_thin_boxes(env, dims):  # noqa: F811
    """Boxes of one- and two-dimensional grids, whose last extents are 1, and others walked along another axis."""
    torch, cr = env
    flat, x, t, mask = random_case(cr, sum(dims) + 1, dims, 3)
    mask[0, 0, 0] = 1
    out, loss, g = cr.ConvNet.check_f64(dims, flat, x, t, mask)
    Ws, bs = unpack(flat)
    ref, loss_ref, dWs, dbs = oracle_all(x, Ws, bs, t, mask)
    assert np.linalg.norm(out - ref) <= 1e-10 * np.linalg.norm(ref)
    close(g, dWs, dbs, 1e-10)


def test_infinite_input_behind_dead_units(env):  # noqa: F811
    """Every unit that sees the infinite input is dead: its gradient is zero and the input adds
    nothing, as a large finite one does."""
    torch, cr = env
    dims, B = (3, 4, 40), 2
    flat, x, t, mask = random_case(cr, 5, dims, B)
    W0 = flat[: 16 * 2 * 27].reshape(16, 2, 27)
    W0[:, 0] = -0.05 - np.abs(W0[:, 0])
    grads = []
    for big in (1e6, np.inf):
        x[1, 0, 1, 2, 36] = big
        grads.append(cr.ConvNet.check_f64(dims, flat, x, t, mask)[2])
    x[1, 0, 1, 2, 36] = 1e6
    Ws, bs = unpack(flat)
    _, _, dWs, dbs = oracle_all(x, Ws, bs, t, mask)
    for g in grads:
        close(g, dWs, dbs, 1e-10)
