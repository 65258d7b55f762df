"""Output layer with weights that have overflowed: a neighbour beyond a closed
face takes no part in the sum, so an infinite or NaN weight that only meets such
neighbours changes nothing."""
import numpy as np
import pytest

import paper_1710_09421_gb300 as E
from paper_1710_09421_gb300 import warmstart

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_weights_beyond_closed_faces_do_not_matter(axis, bad):
    dims, periodic = [9, 7, 5], [1, 1, 1]
    dims[axis], periodic[axis] = 1, 0  # every neighbour along this axis is beyond a face
    x = np.random.default_rng(2).standard_normal((2,) + tuple(dims[::-1])).astype(np.float32)
    w = warmstart.init_params(3).astype(np.float32)
    w4 = w[-(16 * 27 + 1):-1].reshape(16, 3, 3, 3)  # [channel][dz][dy][dx]
    off = np.moveaxis(w4, 3 - axis, 1)
    off[:, [0, 2]] = 0.0
    y = E.ekl_net_eval(dims, periodic, x, w)
    off[:, [0, 2]] = bad
    assert np.isfinite(y).all() and np.ptp(y) > 0
    assert np.array_equal(E.ekl_net_eval(dims, periodic, x, w), y)
