"""Batches in which some replicas have the fluctuating term and some do not: one
launch serves both, and each replica evolves as on its own handle."""
import numpy as np
import pytest

import paper_1710_09421_gb300 as E
from paper_1710_09421_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f64", "f32", "fp16"])
@pytest.mark.parametrize("masses", [(1e-5, 0.0, 1e-6), (0.0, 0.0, 1e-6)])
def test_replicas_with_and_without_fluctuations(precision, masses):
    wls = [W.small_pore(nx=16 + 4 * r, ny=16, nz=20, membrane=(8, 11), radius=3.0, n_beads=2 * r, seed_noise=3 + r,
                        precision=precision).replace(fluct_mass=m, poisson_fixed_iter=20)
           for r, m in enumerate(masses)]
    batch = E.Batch(wls)
    assert batch.step(6) >= 0
    for r, wl in enumerate(wls):
        sim = E.Simulation(wl)
        assert sim.step(6) >= 0
        a, b = sim.get_state(), batch.reps[r].get_state()
        sim.close()
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]), r
    batch.close()
