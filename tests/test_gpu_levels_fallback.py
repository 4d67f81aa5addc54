"""Credible levels in the smaller clusters that take over where one of sixteen CTAs cannot be
placed: against numpy at the edges of each cluster's stride."""
import numpy as np
import pytest

from gpu_common import m, torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_ctas", [16, 8, 1])
@pytest.mark.parametrize("n", [1, 513, 8 * 512 + 1, 4 * 8 * 512 - 1, 100_003])
def test_levels_in_smaller_clusters(m, torch, n, max_ctas):  # noqa: F811
    rng = np.random.default_rng(n)
    theta, w, ref = rng.normal(size=(3, n)), rng.exponential(size=n), rng.normal(size=3)
    w[1::11], theta[2, ::3], ref[2] = 0.0, 0.5, 0.5
    want = ((theta < ref[:, None]) @ w + 0.5 * ((theta == ref[:, None]) @ w)) / w.sum()
    out = torch.empty(3, dtype=torch.float64, device="cuda")
    m.mbis_debug_credible_levels(n, torch.tensor(theta, device="cuda"), torch.tensor(w, device="cuda"), ref, out, max_ctas)
    # sums of at most 1e5 FP64 terms of one sign: far below 1e-12
    assert np.abs(out.cpu().numpy() - want).max() <= 1e-12
