"""A sample whose phase terms leave the fixed-point range (beyond 2^40 turns) is summed in FP64; the
samples that share its tile keep their bits."""
import numpy as np
import pytest

import workloads
from gpu_common import m, torch  # noqa: F401
from test_gpu_fp64 import SKY, SLOTS, build, device, samples

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ids", [SLOTS, SLOTS + SKY])
@pytest.mark.parametrize("marg", [workloads.MARG_PHASE, workloads.MARG_PHASE | workloads.MARG_DISTANCE])
def test_neighbours_of_a_far_sample(m, torch, ids, marg):  # noqa: F811
    ev, th, rng = build(2049, 0.25, 2, marg, (30.0, 25.0), 9)
    full = samples(ev, th, ids, 70, rng)
    want = device(m, torch, ev, th, ids, marg, full)
    far = np.array([10, 33, 69])
    full[far, workloads.TC] = [1e12, -3e13, 1e300]
    got = device(m, torch, ev, th, ids, marg, full)
    rest = np.delete(np.arange(70), far)
    assert np.array_equal(got[rest], want[rest], equal_nan=True)
    assert np.all(np.isfinite(got[far[:2]]))
