"""Training batches that do not go through the network in one pass: split passes
add up to the same parameters and losses, and a batch whose buffers exceed the
device is taken in several passes instead of refused."""
import ctypes as C

import numpy as np
import pytest

import paper_1710_09421_gb300 as E
from paper_1710_09421_gb300 import warmstart

pytestmark = pytest.mark.gpu


def _in_passes(dims, periodic, x, t, mask, w, iters, batch, lr, seed, pass_bytes):
    f = E.load().ekl_net_train_in_passes
    vp = C.c_void_p
    f.argtypes = [C.c_int32, vp, vp, vp, vp, vp, vp, C.c_int32, C.c_int32, C.c_float, C.c_uint64, vp, C.c_uint64]
    p = lambda a: None if a is None else a.ctypes.data_as(vp)
    d, per, w, curve = np.asarray(dims, np.int32), np.asarray(periodic, np.int32), w.copy(), np.zeros(iters, np.float32)
    assert f(len(x), p(d), p(per), p(x), p(t), p(mask), p(w), iters, batch, lr, seed, p(curve), pass_bytes) == 0
    return w, curve


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("dims", [(18, 9, 6), (3, 2, 2)])  # two and one runs of 512 nodes
def test_split_passes_equal_one_pass(dims, masked):
    rng = np.random.default_rng(4)
    shape = dims[::-1]
    x, t = rng.standard_normal((3, 2) + shape).astype(np.float32), rng.standard_normal((3,) + shape).astype(np.float32)
    mask = (rng.random(shape) < 0.7).astype(np.uint8) if masked else None
    w = warmstart.init_params(1).astype(np.float32)
    iters, batch = 1100, 5  # several uploads of sample numbers (4096) and read-backs of losses (512)
    w0, c0 = E.ekl_net_train_grid(dims, (1, 0, 1), x, t, mask, w, iters, batch, 1e-3, 9)
    assert np.isfinite(c0).all() and c0[-1] < c0[0]
    n = dims[0] * dims[1] * dims[2]
    sample = 4 * 15169 * -(-n // 512) + 180 * n + 4096  # about one sample's buffers
    for pass_bytes in (2 * sample, sample, 0):
        w1, c1 = _in_passes(dims, (1, 0, 1), x, t, mask, w, iters, batch, 1e-3, 9, pass_bytes)
        assert np.array_equal(w1, w0), pass_bytes  # the samples' gradients are added in the same order
        # FP64 sums in another order, rounded to FP32
        assert np.abs(c1 - c0).max() <= 2.0 ** -23 * np.abs(c0).max(), pass_bytes


def test_batch_larger_than_the_device_is_not_refused():
    """Five million samples ask for 300 GB of partials at once.  With all
    parameters zero the output is zero, so the loss is the mean square of the drawn
    targets and only the last bias moves, by lr g / (|g| + 1e-8), g = -2 mean(t)."""
    dims, ns, batch, lr, seed = (1, 1, 1), 4, 5_000_000, 1e-3, 5
    c = np.array([1.0, 2.0, 4.0, 7.0]) * 1e-8
    x = np.random.default_rng(0).standard_normal((ns, 2, 1, 1, 1)).astype(np.float32)
    t = np.broadcast_to(c.reshape(ns, 1, 1, 1), (ns, 1, 1, 1)).astype(np.float32)
    w, curve = E.ekl_net_train_grid(dims, (1, 1, 1), x, t, None, np.zeros(E.EKL_NET_PARAMS, np.float32), 1, batch, lr,
                                    seed)
    st = (np.uint64(seed) + np.uint64(0x9E3779B97F4A7C15) * np.arange(1, batch + 1, dtype=np.uint64))
    z = (st ^ (st >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    share = np.bincount(((z ^ (z >> np.uint64(31))) % np.uint64(ns)).astype(int), minlength=ns) / batch
    assert abs(curve[0] / (share * c ** 2).sum() - 1.0) < 1e-5  # FP32 squares, FP64 sums
    g = 2.0 * (share * c).sum()
    # FP32 sums of one term per sample, one after the other: at most batch 2^-24 = 0.3
    # of g; a pass that is lost (of 72) or counted alone leaves no more than g / 70
    lo, hi = (lr * f * g / (f * g + 1e-8) for f in (0.7, 1.3))
    assert lo < w[-1] < hi and not w[:-1].any()
