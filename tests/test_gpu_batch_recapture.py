"""A batch whose events' proposals or metrics move between its steps captures its graph again for
each: every step must equal the single-event entry points on the moved proposals, bit for bit."""
import numpy as np
import pytest

import workloads
from gpu_common import m, torch, set_metric  # noqa: F401
from test_gpu_batch import build

pytestmark = pytest.mark.gpu


def test_steps_after_moved_proposals(m, torch):  # noqa: F811
    evs = build(workloads.uneven_batch()[:3], m, [500, 4096, 700])
    pick = [evs[i % 3] for i in range(10)]  # more entries than branches
    ns = [e["w"].n_samples + i for i, e in enumerate(pick)]
    b = m.mbis_batch_create([e["ctx"] for e in pick], ns, [5 + i for i in range(10)])
    try:
        for step in range(6):
            e = evs[step % 3]
            if step == 4:
                set_metric(m, e["ctx"], e["prop"])
            elif step:
                mean = e["prop"]["mean"] + 0.1 * step * np.diag(np.asarray(e["prop"]["chol"]))
                m.mbis_set_proposal(e["ctx"], mean, e["prop"]["chol"], 1.0 + 0.1 * step)
            sums = m.mbis_batch_step(b, step, 10)
            for i, e in enumerate(pick):
                n, P = ns[i], len(e["prop"]["ids"])
                th = torch.empty((P, n), dtype=torch.float64, device="cuda")
                lq, lp, ll = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(3))
                m.mbis_draw(e["ctx"], 5 + i, step * n, n, th, lq, lp)
                m.mbis_loglike(e["ctx"], n, th, ll)
                ref = m.mbis_reduce(e["ctx"], n, ll, lp, lq, None, 0)
                for k in ("ess", "log_z", "max_logw", "s1", "s2", "n"):
                    assert sums[i][k] == ref[k], (step, i, k)
    finally:
        m.mbis_batch_destroy(b)
        for e in evs:
            m.mbis_destroy(e["ctx"])
