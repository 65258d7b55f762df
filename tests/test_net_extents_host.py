"""The warm-start network's entry points refuse grids that their kernels cannot
index before any CUDA work (no GPU needed): an empty or negative extent (the
splits into tiles divide by it) and more than 2^30 nodes."""
import ctypes as C

import numpy as np
import pytest

import paper_1710_09421_gb300 as E


@pytest.mark.parametrize("dims", [(0, 4, 4), (4, 0, 4), (4, 4, 0), (0, 0, 0), (-1, 4, 4), (-2, -2, 4), (4, 4, -1),
                                  (2048, 2048, 2048), (1 << 30, 2, 1), (1 << 16, 1 << 16, 1 << 16)])
def test_grids_that_cannot_be_indexed_are_refused(dims):
    L = E.load()
    d, per = np.asarray(dims, np.int32), np.zeros(3, np.int32)
    buf = np.zeros(E.EKL_NET_PARAMS, np.float32)  # never read
    p, loss = (lambda a: a.ctypes.data_as(C.c_void_p)), C.c_double(0)
    for rc in (L.ekl_net_eval(p(d), p(per), p(buf), p(buf), p(buf)),
               L.ekl_net_loss_grad(p(d), p(per), p(buf), p(buf), None, p(buf), C.byref(loss), p(buf)),
               L.ekl_net_train_grid(1, p(d), p(per), p(buf), p(buf), None, p(buf), 1, 1, 1e-3, 0, None),
               L.ekl_net_train(1, p(d), p(buf), p(buf), None, p(buf), 1, 1, 1e-3, 0, None)):
        assert rc == E.EKL_ERR_ARG
        assert b"extent" in L.ekl_last_error() or b"too large" in L.ekl_last_error()
