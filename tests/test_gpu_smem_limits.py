"""A kernel's shared-memory limit is shared by every handle of the process:
creating a handle or a batch whose coarse levels need little of it must not take
it away from one that needs more."""
import pytest

import paper_1710_09421_gb300 as E
from paper_1710_09421_gb300 import workloads as W
from helpers import box

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [W.FLAG_POISSON_MG, W.FLAG_POISSON_MG | W.FLAG_POISSON_MG_SINGLE, 0])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_a_smaller_handle_leaves_the_limit(flags, precision):
    kw = dict(precision=precision, flags=flags, E_app=(1e-3, 0.0, 0.0))
    large = E.Simulation(box(36, 28, 60, **kw))  # 7560 cells at the coarsest level
    assert large.step(1) >= 0
    small = E.Simulation(box(16, 16, 16, **kw))
    assert small.step(1) >= 0 and large.step(1) >= 0
    small.close()
    large.close()


@pytest.mark.parametrize("flags", [W.FLAG_POISSON_MG, W.FLAG_POISSON_MG | W.FLAG_POISSON_MG_SINGLE])
def test_a_smaller_batch_leaves_the_limit(flags):
    kw = dict(precision="f32", flags=flags)
    large = E.Batch([box(36, 28, 60, **kw), box(36, 28, 60, **kw)])
    assert large.step(1) >= 0
    small = E.Batch([box(16, 16, 16, **kw)])
    assert small.step(1) >= 0 and large.step(1) >= 0
    small.close()
    large.close()
