"""The ordered weight reduction of the ESS loop's refit batches where its shape changes: less
than a warp, a CTA and one more, the serial sum's groups of CTAs, and more samples than the grid
has threads.  The loop's own log likelihoods, priors and densities give the weights in numpy."""
import numpy as np
import pytest

import workloads
from gpu_common import m, torch  # noqa: F401
from test_gpu_batch import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [17, 256, 257, 16 * 256 + 1, 17 * 256, 608 * 256 + 3])
def test_weights_of_a_refit_batch(m, torch, n):  # noqa: F811
    e = build(workloads.uneven_batch()[:1], m, [n])[0]
    P = len(e["prop"]["ids"])
    th = torch.empty((P, n), dtype=torch.float64, device="cuda")
    lq, lp, ll, w = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(4))
    try:
        s, drawn, _ = m.mbis_run_to_ess(e["ctx"], th, lq, lp, ll, w, 1e12, n, n, 3, refine=1)
        torch.cuda.synchronize()
    finally:
        m.mbis_destroy(e["ctx"])
    assert drawn == n
    lw = (ll + lp - lq).cpu().numpy()
    want = np.exp(lw - lw.max())
    want /= want.sum()
    # a sum of n terms of one sign in any order is within n u, an exponential and the scaling
    # within a few u more
    assert np.all(np.abs(w.cpu().numpy() - want) <= (n + 16) * 2.0 ** -53 * want + 1e-300)
