"""The tiled SOR kernel against the global-memory one at the shapes where its
index work can go wrong: rows of odd length, tiles thinner than two halos,
tiles that wrap onto themselves, more nodes per thread than it keeps in
registers, closed sides.  Both do the same node updates in the same schedule,
so potentials and sweep counts agree bit for bit."""
import numpy as np
import pytest

import paper_1710_09421_gb300 as E
from paper_1710_09421_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("dims,periodic", [
    ((40, 13, 13), (1, 0, 0)),   # one tile of 13 x 13 rows: 4420 red nodes
    ((33, 24, 20), (0, 1, 1)),   # odd rows
    ((16, 4, 6), (1, 1, 1)),     # a tile's halo reaches its own rows
    ((26, 60, 84), (1, 1, 0)),   # tiles with an interior beyond the rim, closed z
    ((3, 8, 10), (0, 1, 1)),     # rows of two pairs
])
def test_tiled_sor_equals_global(dims, periodic, precision):
    nx, ny, nz = dims
    rng = np.random.default_rng(7)
    solid = np.zeros((nz, ny, nx), np.uint8)
    solid[nz // 2, : ny // 2, : (nx + 1) // 2] = 1
    n = W.ion_densities(solid, 0.01, 1.0, 0.0, 3e-3, int(rng.integers(1 << 30)))
    wl = W.Workload(name="box", nx=nx, ny=ny, nz=nz, periodic=periodic, solid=solid, surface_charge=None, n_init=n,
                    n_ref=(1.0, 0.01, 0.01), E_app=(1e-3, 0.0, 2e-3), precision=precision, poisson_fixed_iter=7,
                    rho_jacobi=0.98)
    out = []
    for flags in (0, W.FLAG_POISSON_GLOBAL):
        sim = E.Simulation(wl.replace(flags=flags))
        sim.step(3)
        f, phi, _ = sim.get_state()
        out.append((f, phi, sim.stats()["poisson_sweeps"]))
        sim.close()
    assert out[0][2] == out[1][2] == 21
    assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][0], out[1][0])
    assert np.abs(out[0][1]).max() > 0
