"""Retraining at the sizes where its kernels change shape, against the oracle.

Rows: below, at and beyond multiples of 16 (a row block), 512 and 2048 (where
the gradients' rows are cut in more parts) and 152 x 16 (more row blocks than
SMs).  Bounds: those that the gradients, targets and losses of the same
operands are held to at the ordinary sizes."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu

swig = pytest.importorskip("paper_2607_28265_gb300.swig")


@pytest.fixture(scope="module")
def ctx():
    c = swig.Context(0)
    yield c
    c.close()


def _live(n, d, seed):
    rng = np.random.default_rng(seed)
    t = rng.random(n)
    u = 0.5 + 0.05 * rng.standard_normal((n, d)) + 0.1 * np.outer(t, np.arange(d) % 3 - 1)
    u[:, 0] = 0.2 + 0.6 * t
    return np.clip(u, 0.0, 1.0)


@pytest.mark.parametrize("n,d", [(1, 13), (15, 3), (16, 13), (17, 1), (511, 4), (512, 12), (2047, 2), (2048, 12),
                                 (2433, 9)])
def test_gradient_and_outputs(ctx, n, d):
    rng = np.random.default_rng(n)
    params = mlp.init_params(n)
    x = np.zeros((n, mlp.D_IN))
    x[:, :d] = rng.standard_normal((n, d))
    tdir = np.zeros((n, mlp.D_IN), np.float32)
    tdir[:, :d] = rng.standard_normal((n, d))
    tdir /= np.linalg.norm(tdir, axis=1, keepdims=True)
    tls = np.zeros((n, mlp.D_IN), np.float32)
    tls[:, :d] = -2.0 + 0.3 * rng.standard_normal((n, d))
    cache = mlp.forward(params, x, bf16=True)
    want_loss, dO = mlp.loss_and_dout(cache["O"], tdir, tls, d)
    want = mlp.backward(params, cache, dO, bf16=True)
    out = ctx.mlp_forward(params, x)
    assert np.max(np.abs(out - cache["O"])) <= 2e-3 * np.max(np.abs(cache["O"]))
    loss, g = ctx.mlp_loss_grad(params, x, tdir, tls, d)
    assert abs(loss - want_loss) <= 1e-4 * abs(want_loss)
    offs = np.cumsum([0] + [int(np.prod(s)) for s in mlp.SHAPES])
    for a, b in zip(offs[:-1], offs[1:]):
        assert np.max(np.abs(g[a:b] - want[a:b])) <= 1e-2 * np.max(np.abs(want[a:b]))


@pytest.mark.parametrize("n,d,twins", [(28, 13, 0), (33, 3, 0), (150, 12, 0), (900, 5, 0), (300, 4, 200)])
def test_neighbours_and_widths(ctx, n, d, twins):
    """FP32 finds the candidates, FP64 decides: the oracle's neighbours in the
    oracle's order, also with more equal points than there is room for."""
    live = _live(n, d, n)
    live[:twins] = live[0]
    _, tls, nbr = ctx.mlp_targets(live)
    _, want_ls, want_nbr, _ = mlp.local_pca_targets(live, details=True)
    assert np.array_equal(nbr[:, :2 * d], np.asarray(want_nbr)[:, :2 * d])
    ok = np.isfinite(want_ls)
    assert np.all(np.abs(tls - want_ls)[ok] <= 1e-6 * np.abs(want_ls[ok]) + 1e-6)
