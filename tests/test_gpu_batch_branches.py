"""A batch step runs its events' draws and reductions on up to eight branches of its graph.
More entries than branches, with contexts that appear several times (their reductions share
one scratch): every summary must equal the one of the single-event entry points on the same
draws, bit for bit, step after step."""
import pytest

import workloads
from gpu_common import m, torch  # noqa: F401
from test_gpu_batch import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("entries", [1, 2, 8, 9, 19])
def test_branches_and_shared_contexts(m, torch, entries):
    evs = build(workloads.uneven_batch()[:3], m, [129, 4096, 700])
    pick = [evs[i % 3 if i % 4 else 0] for i in range(entries)]
    ns = [e["w"].n_samples + 7 * i for i, e in enumerate(pick)]
    seeds = [e["spec"].draw_seed + i for i, e in enumerate(pick)]
    b = m.mbis_batch_create([e["ctx"] for e in pick], ns, seeds)
    try:
        for step in (0, 3, 0):
            sums = m.mbis_batch_step(b, step, entries)
            for i, e in enumerate(pick):
                n, P = ns[i], len(e["prop"]["ids"])
                th = torch.empty((P, n), dtype=torch.float64, device="cuda")
                lq, lp, ll = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(3))
                m.mbis_draw(e["ctx"], seeds[i], step * n, n, th, lq, lp)
                m.mbis_loglike(e["ctx"], n, th, ll)
                ref = m.mbis_reduce(e["ctx"], n, ll, lp, lq, None, 0)
                for k in ("ess", "log_z", "max_logw", "s1", "s2", "n"):
                    assert sums[i][k] == ref[k], (entries, step, i, k)
    finally:
        m.mbis_batch_destroy(b)
        for e in evs:
            m.mbis_destroy(e["ctx"])
