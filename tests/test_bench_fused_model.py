"""bench.py's byte and launch counts of the multigrid solve that takes two half
sweeps per launch, and the rule that tells it from the other form (no GPU)."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402
from paper_1710_09421_gb300 import workloads as W  # noqa: E402


class _Box:
    def __init__(self, nx, ny, nz, flags=W.FLAG_POISSON_MG):
        self.nx, self.ny, self.nz, self.n_nodes, self.flags = nx, ny, nz, nx * ny * nz, flags


def test_bytes_and_launches():
    # four fused passes, r.z, p/q, update, coarse levels
    assert bench.MG_FUSED_BYTES_PER_ITER == 108.5 and bench.MG_FUSED_BYTES_PER_SOLVE == 57
    huge = _Box(256, 256, 512)
    # pre-smoothing, restriction, coarse launch, two passes, r.z, p/q, update, mid, residual, end; level 1's eight
    assert bench.mg_split_kernels_per_iter(huge, fused=True) == 11 + 8
    assert bench.mg_split_kernels_per_iter(huge) == 14 + 8
    assert bench.mg_split_kernels_per_iter(_Box(64, 64, 128)) == 14


def test_which_lattices_take_two_half_sweeps():
    for dims, fused in (((256, 256, 512), True), ((128, 128, 256), True), ((64, 64, 128), False),
                        ((100, 192, 192), True), ((102, 192, 192), False), ((96, 192, 192), False)):
        assert bench.mg_fused(W, _Box(*dims)) == fused, dims
    assert not bench.mg_fused(W, _Box(256, 256, 512, W.FLAG_POISSON_MG | W.FLAG_POISSON_MG_SINGLE))
