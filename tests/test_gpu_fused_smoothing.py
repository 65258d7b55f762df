"""The lattice smoothing that takes two half sweeps per launch (lattices whose
solve does not stay in L2) against the same solve in one cooperative launch
(EKL_POISSON_MG_SINGLE), whose passes take one half sweep at a time: the
updates, their rounding and the order of every sum are the same, so the
potential, the iteration counts and the residuals agree bit for bit.  Shapes:
whole rows, x-segments (rows too long for a tile), rows of pieces of eight and
of four nodes, ragged last tiles, closed sides with an odd extent."""
import numpy as np
import pytest

import paper_1710_09421_gb300 as E
from paper_1710_09421_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MG = W.FLAG_POISSON_MG


def _box(nx, ny, nz, periodic, precision):
    rng = np.random.default_rng(nx + ny)
    solid = np.zeros((nz, ny, nx), np.uint8)
    solid[nz // 3: nz // 3 + 5, :, : nx // 2] = 1
    solid[:, ny // 2, 3: nx // 3] = 1
    n = W.ion_densities(solid, 0.01, 1.0, 0.0, 3e-3, int(rng.integers(1 << 30)))
    return W.Workload(name="box", nx=nx, ny=ny, nz=nz, periodic=periodic, solid=solid, surface_charge=None, n_init=n,
                      n_ref=(1.0, 0.01, 0.01), E_app=(1e-3, 0.0, 2e-3), precision=precision, poisson_tol=1e-8)


@pytest.mark.parametrize("dims,periodic,precision", [
    ((256, 128, 128), (1, 1, 1), "f32"),   # whole rows of 32 threads
    ((640, 64, 128), (1, 1, 1), "f32"),     # x-segments, the last one ragged
    ((180, 152, 152), (0, 0, 0), "f32"),   # pieces of four nodes (closed: an odd extent halves)
    ((96, 207, 209), (1, 0, 0), "f32"),    # odd closed extents
    ((160, 256, 96), (0, 1, 0), "f64"),   # closed rows, FP64
])
def test_fused_smoothing_equals_single_launch(dims, periodic, precision):
    wl = _box(*dims, periodic, precision)
    assert wl.n_nodes * 37 > 126 << 20  # larger than L2: the fused form
    out = []
    for flags in (MG, MG | W.FLAG_POISSON_MG_SINGLE):
        sim = E.Simulation(wl.replace(flags=flags))
        its = []
        for _ in range(2):
            assert sim.step(1) >= 0
            st = sim.stats()
            its.append((st["poisson_iters"], st["poisson_res"]))
        out.append((sim.fields(("n", "phi")), its))
        sim.close()
    (fa, ia), (fb, ib) = out
    assert ia == ib
    for k in ("n", "phi"):
        assert np.array_equal(fa[k], fb[k]), k


@pytest.mark.parametrize("boxes", [
    [(96, 96, 192), (128, 96, 128), (48, 48, 192)],   # pieces of eight nodes
    [(100, 96, 192), (128, 96, 128), (48, 48, 192)],  # of four for all
])
def test_batch_fused_smoothing_equals_cooperative(boxes):
    """The same for a batch whose replicas together exceed L2: the launches of
    two half sweeps over all replicas and one cooperative launch (schedule 2:
    the same blocks per replica) return the same bits."""
    wls = [_box(*d, (0, 1, 1), "f32") for d in boxes]
    assert sum(w.n_nodes for w in wls) * 37 > 126 << 20
    a = E.Batch([w.replace(flags=MG) for w in wls])
    b = E.Batch([w.replace(flags=MG | W.FLAG_POISSON_MG_SINGLE) for w in wls])
    a.set_schedule(2)
    b.set_schedule(2)
    for _ in range(2):
        assert a.step(1) >= 0 and b.step(1) >= 0
        for r in range(len(wls)):
            sa, sb = a.reps[r].stats(), b.reps[r].stats()
            assert sa["poisson_iters"] == sb["poisson_iters"] > 0 and sa["poisson_res"] == sb["poisson_res"], r
    for r in range(len(wls)):
        fa, fb = a.reps[r].fields(("n", "phi")), b.reps[r].fields(("n", "phi"))
        assert np.array_equal(fa["n"], fb["n"]) and np.array_equal(fa["phi"], fb["phi"]), r
    a.close()
    b.close()


@pytest.mark.parametrize("dims,periodic", [
    ((40, 24, 36), (1, 1, 1)),   # 4320 cells: positions kept in registers
    ((36, 28, 60), (1, 1, 1)),   # 7560 cells: positions formed in every sweep
    ((27, 22, 20), (0, 0, 1)),   # odd closed rows
    ((25, 19, 21), (0, 0, 0)),   # odd in every extent
])
def test_coarsest_level_of_block_zero_meets_tolerance(dims, periodic):
    """Coarsest levels smoothed by one block: the converged potential meets the tolerance under the oracle's
    operator and source."""
    import oracle

    nx, ny, nz = dims
    wl = _box(nx, ny, nz, periodic, "f64").replace(poisson_tol=1e-9, flags=MG)
    sim = E.Simulation(wl)
    ref = oracle.Sim(wl.replace(poisson_tol=1e-13), threads=8)
    assert sim.step(1) >= 0 and ref.step(1) >= 0
    _, phi, _ = sim.get_state()
    assert ref.poisson_residual(ref.last_rho(), phi) <= 1e-9 * 1.001
    sim.close()
