"""Warm-start network on grids whose extents fall on the edges of the
kernels' tiles (30 nodes along x, 128 rows per plane, 2 planes) and of the
weight gradient's 16- and 512-node runs: loss and every parameter block against
the FP64 oracle, and a training batch of several samples against the oracle's
gradient and a plain Adam step."""
import numpy as np
import pytest

import paper_1710_09421_gb300 as E
from oracle import net

pytestmark = pytest.mark.gpu


def _inputs(seed, shape, ns=1):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((ns, 2) + shape).astype(np.float32)
    t = rng.standard_normal((ns,) + shape).astype(np.float32)
    w = (net.init_params(seed) + 0.02 * rng.standard_normal(net.n_params())).astype(np.float32)
    return x, t, w


@pytest.mark.parametrize("dims,periodic", [((30, 5, 4), (1, 1, 1)), ((31, 6, 5), (0, 1, 0)), ((61, 3, 2), (1, 0, 1)),
                                           ((16, 7, 8), (0, 0, 0)), ((17, 13, 9), (1, 1, 0)), ((2, 45, 3), (1, 1, 1))])
def test_gradient_on_tile_edges(dims, periodic):
    nx, ny, nz = dims
    x, t, w = _inputs(nx, (nz, ny, nx))
    mask = np.ones((nz, ny, nx), np.uint8)
    mask[0, 0, : nx // 2] = 0
    loss, grad = E.ekl_net_loss_grad(dims, periodic, x[0], t[0], mask, w)
    rl, rg = net.loss_grad(x[0].astype(np.float64), t[0].astype(np.float64), mask, w.astype(np.float64), periodic)
    # BF16 activations and weights: the bounds of the network's other gradient test
    assert abs(loss - rl) / rl < 2e-2
    o = 0
    for ci, co in zip(net.CHANNELS[:-1], net.CHANNELS[1:]):
        for n in (co * ci * 27, co):
            a, b = grad[o:o + n], rg[o:o + n]
            assert np.linalg.norm(a - b) / np.linalg.norm(b) < 5e-2, (ci, co, n)
            o += n


def test_training_batch_is_the_mean_of_its_samples():
    """One Adam step from zero moments moves every parameter by lr g / (|g| +
    eps'), so the sign pattern and the loss show the batch's mean gradient."""
    dims, periodic, ns, lr = (18, 9, 6), (1, 1, 0), 5, 1e-3
    x, t, w = _inputs(7, dims[::-1], ns)
    w1, curve = E.ekl_net_train_grid(dims, periodic, x, t, None, w, 1, batch=4, lr=lr, seed=3)
    st, pick = 3, []
    for _ in range(4):
        st = (st + 0x9E3779B97F4A7C15) % 2 ** 64
        z = ((st ^ (st >> 30)) * 0xBF58476D1CE4E5B9) % 2 ** 64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) % 2 ** 64
        pick.append((z ^ (z >> 31)) % ns)
    mask = np.ones(dims[::-1])
    out = [net.loss_grad(x[s].astype(np.float64), t[s].astype(np.float64), mask, w.astype(np.float64), periodic)
           for s in pick]
    loss, g = np.mean([o[0] for o in out]), np.mean([o[1] for o in out], axis=0)
    assert abs(curve[0] - loss) / loss < 2e-2
    big = np.abs(g) > 0.2 * np.sqrt(np.mean(g ** 2))  # away from the BF16 error of the gradient
    step = (w.astype(np.float64) - w1)[big] / lr
    assert np.mean(np.sign(step) == np.sign(g[big])) > 0.99
    assert np.abs(np.abs(step) - 1.0).max() < 1e-2
