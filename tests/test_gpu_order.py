"""The work order's edges, through entry points whose results do not depend on it: keys counted
in shared memory and, beyond, per warp (a 2-bin key per 128k-bin grid); sample counts around a
CTA, the grid and the samples a thread keeps.  A wrong order (a slot lost or doubled) leaves
samples of the output untouched or evaluates others twice."""
import numpy as np
import pytest

import workloads
from oracle.events import make_event, make_proposal
from gpu_common import m, torch, gpu_context, set_metric  # noqa: F401

pytestmark = pytest.mark.gpu

GRID = 304 * 512


@pytest.fixture(scope="module", params=[0.125, 1 / 128])
def event(m, request):  # noqa: F811
    w = workloads.scaled(workloads.bbh_pp_population(1), n_events=1, f_hi=512.0 if request.param == 0.125 else 420.0)
    w.df = request.param
    ev, th, _ = make_event(w, w.events[0])
    ctx = gpu_context(m, ev, w, w.events[0], th, m.MIXED)
    prop = make_proposal(ev, w, th)
    prop["lo"] = np.maximum(prop["lo"], [0.1 * th[0], 1.0, -0.9, -0.9, -1.0])  # a wide metric: keep the box physical
    set_metric(m, ctx, prop)
    yield ctx, 5
    m.mbis_destroy(ctx)


@pytest.mark.parametrize("n", [4096, 4097, GRID - 1, GRID + 1, 8 * GRID + 513])
def test_every_sample_is_evaluated_once(m, torch, event, n):  # noqa: F811
    ctx, P = event
    theta = torch.empty((P, n), dtype=torch.float64, device="cuda")
    m.mbis_draw(ctx, 3, 0, n, theta)
    out = torch.full((n,), 1e300, dtype=torch.float64, device="cuda")
    m.mbis_loglike(ctx, n, theta, out)
    # pieces below 4096 samples are evaluated in the order given
    idx = np.unique(np.concatenate([np.arange(2000), np.arange(n - 2000, n)]))
    for part in np.array_split(idx, 2):
        sub = theta[:, torch.tensor(part, device="cuda")].contiguous()
        ref = torch.empty(len(part), dtype=torch.float64, device="cuda")
        m.mbis_loglike(ctx, len(part), sub, ref)
        assert torch.equal(out[torch.tensor(part, device="cuda")], ref)
    assert not bool((out == 1e300).any())
