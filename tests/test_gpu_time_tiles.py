"""The time-marginalised kernel's tiles of 32, 64 and 128 samples: a sample's log L does not
depend on the tile it is evaluated in (bit for bit), for one to four detector rows, at the edges
of the rule and with part-filled tiles; and matches the oracle on the smallest."""
import numpy as np
import pytest

import oracle
import workloads
from oracle.events import make_event, make_proposal
from gpu_common import m, torch, gpu_context, set_metric, compare_loglike  # noqa: F401

pytestmark = pytest.mark.gpu

SMS = 152
EDGES = [1, 31, 33, 32 * SMS, 32 * SMS + 1, 64 * SMS, 64 * SMS + 1]


@pytest.mark.parametrize("dets", [["H1"], ["H1", "L1"], ["H1", "L1", "V1"]])
@pytest.mark.parametrize("sky", [True, False])
def test_tiles_agree_bit_for_bit(m, torch, dets, sky):  # noqa: F811
    w = workloads.scaled(workloads.bbh_population(1), n_events=1, f_hi=200.0)
    w.detectors = dets
    if not sky:  # one folded row
        w.sampled = [s for s in w.sampled if s not in (workloads.RA, workloads.DEC, workloads.PSI, workloads.IOTA)]
    ev, th, _ = make_event(w, w.events[0])
    prop = make_proposal(ev, w, th)
    prop["lo"] = np.where(np.isin(prop["ids"], [0, 1, 8]), np.maximum(prop["lo"], 0.1), prop["lo"])
    ctx = gpu_context(m, ev, w, w.events[0], th, m.MIXED)
    try:
        set_metric(m, ctx, prop)
        P, n = len(prop["ids"]), EDGES[-1]
        theta = torch.empty((P, n), dtype=torch.float64, device="cuda")
        lp = torch.empty(n, dtype=torch.float64, device="cuda")
        m.mbis_draw(ctx, 9, 0, n, theta, None, lp)
        ref = torch.empty(n, dtype=torch.float64, device="cuda")
        m.mbis_loglike(ctx, n, theta, ref)  # 128-sample tiles
        for k in EDGES[:-1]:
            out = torch.full((k,), 1e300, dtype=torch.float64, device="cuda")
            m.mbis_loglike(ctx, k, theta[:, :k].contiguous(), out)
            assert torch.equal(out, ref[:k]), k
        sub = theta[:, :48].cpu().numpy()
        want = oracle.loglike_batch(ev, oracle.full_params(prop["ids"], sub, th))
        compare_loglike(ref[:48].cpu().numpy(), want, lp[:48].cpu().numpy())
    finally:
        m.mbis_destroy(ctx)
