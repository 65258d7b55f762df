"""Bead kernels at the edges of how they share out the beads (a cluster of eight
blocks of sixteen warps, one bead per warp; a counting sort up to 64 beads, a
sorting network above): 1, 8 and 9 beads, 64 and 65, 128 and 129 (several beads per
warp, their noise drawn inside the sub-step) and the most, 256, against the
oracle; and SOR batches whose replicas have their own caps and test intervals
against single handles."""
import numpy as np
import pytest

import oracle
import paper_1710_09421_gb300 as E
from paper_1710_09421_gb300 import workloads as W
from helpers import box, rel

pytestmark = pytest.mark.gpu


def _many_beads(nb, precision, **kw):
    """Chains of up to 37 beads side by side above a wall, close enough for every
    kind of force: bonds, neighbouring chains (1.1 apart), wall nodes (1.05)."""
    n, per_row = 44, 37
    solid = np.zeros((n, n, n), np.uint8)
    solid[10:14] = 1
    k = np.arange(nb)
    row = k // per_row
    rng = np.random.default_rng(nb)
    R = np.stack([3.0 + 0.97 * (k % per_row), 20.0 + 1.1 * (row % 4), 14.05 + 1.1 * (row // 4)], axis=1)
    R += rng.uniform(-0.02, 0.02, R.shape)
    return box(n, n, n, solid=solid, n_init=W.ion_densities(solid, 0.01, 1.0, -0.1 * nb, 1e-4, 3), R=R,
               V=1e-3 * rng.standard_normal(R.shape), charge=np.full(nb, -0.1), chain=row.astype(np.int32),
               E_app=(1e-3, 0.0, 2e-3), precision=precision, poisson_fixed_iter=12, rho_jacobi=0.99, seed=11, **kw)


# FP64: the kernels add in the oracle's order, so a step differs by the rounding of
# what feeds the beads (1e-15), times what three steps of bonds of frequency 3 make
# of it (e^9); FP32: a separation is off by 2^-24 of itself, a force r^-14 of it by
# 14 times that, and the sum of a bond and its neighbours by their cancellation (10)
BOUND = {"f64": 1e-11, "f32": 1e-4}


@pytest.mark.parametrize("bond", [W.BOND_FENE, W.BOND_HARMONIC])
@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("nb", [1, 8, 9, 64, 65, 100, 128, 129, 256])
def test_chains_match_oracle(nb, precision, bond):
    wl = _many_beads(nb, precision, bond_kind=bond)
    sim, ref = E.Simulation(wl), oracle.Sim(wl, threads=8)
    assert sim.step(3) >= 0 and ref.step(3) >= 0
    G, O = sim.fields(), ref.fields()
    sim.close()
    R0 = np.asarray(wl.R)
    for name, g, o in (("R", G["R"] - R0, O["R"] - R0), ("V", G["V"], O["V"])):
        assert np.abs(g - o).max() <= BOUND[precision] * np.abs(o).max(), (name, np.abs(g - o).max() / np.abs(o).max())
    fluid = wl.solid.ravel() == 0
    for a in range(3):  # what the beads spread to the nodes
        assert rel(G["n"][a][fluid], O["n"][a][fluid]) < (1e-5 if precision == "f32" else 1e-12), a


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_batch_of_many_beads_equals_single_runs(precision):
    """Replicas of one launch with no bead, one and several beads per warp; sweeps
    capped by each replica's own maximum (the tolerance is out of reach)."""
    wls = [_many_beads(nb, precision, poisson_tol=1e-30, poisson_max_iter=cap, poisson_check_every=every)
           .replace(poisson_fixed_iter=0) for nb, cap, every in ((256, 13, 1), (40, 31, 5), (129, 22, 3))]
    wls.insert(1, wls[0].replace(R=None, V=None, charge=None, chain=None, poisson_max_iter=9))
    batch = E.Batch(wls)
    assert batch.step(2) >= 0
    for r, wl in enumerate(wls):
        sim = E.Simulation(wl)
        assert sim.step(2) >= 0
        a, b = sim.get_state(), batch.reps[r].get_state()
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]), r
        if wl.R is not None:
            fa, fb = sim.fields(("R", "V")), batch.reps[r].fields(("R", "V"))
            assert np.array_equal(fa["R"], fb["R"]) and np.array_equal(fa["V"], fb["V"]), r
        sa, sb = sim.stats(), batch.reps[r].stats()
        assert sa["poisson_iters"] == sb["poisson_iters"] == wl.poisson_max_iter
        # the same residuals, squared in FP32 (f32) and added in another order
        assert abs(sa["poisson_res"] / sb["poisson_res"] - 1.0) < (1e-5 if precision == "f32" else 1e-12), r
        sim.close()
    batch.close()
