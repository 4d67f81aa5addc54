"""The clustered credible levels where their shape changes: fewer samples than lanes, one CTA,
the cluster's threads and its unrolled stride, with ties at both zeros, NaN samples and
weights that are zero, negative or NaN."""
import numpy as np
import pytest

from gpu_common import m, torch  # noqa: F401

pytestmark = pytest.mark.gpu

CLUSTER = 16 * 512


@pytest.mark.parametrize("n", [1, 31, 512, 513, CLUSTER, CLUSTER + 1, 4 * CLUSTER - 1, 4 * CLUSTER + 1, 300_007])
@pytest.mark.parametrize("P", [1, 3, 16])
def test_levels_at_the_cluster_edges(m, torch, n, P):  # noqa: F811
    rng = np.random.default_rng(100 * P + n)
    theta = rng.normal(size=(P, n))
    theta[0, ::3] = -0.0
    theta[0, 1::5] = 0.0
    theta[P - 1, 2::7] = np.nan
    w = rng.exponential(size=n)
    w[1::11], w[2::13], w[3::17] = 0.0, -1.0, np.nan
    ref = rng.normal(size=P)
    ref[0] = 0.0
    on = w > 0
    tot = w[on].sum()
    want = np.array([(w[on] * (theta[p, on] < ref[p])).sum() + 0.5 * (w[on] * (theta[p, on] == ref[p])).sum()
                     for p in range(P)]) / tot
    out = torch.empty(P, dtype=torch.float64, device="cuda")
    m.mbis_credible_levels(n, torch.tensor(theta, device="cuda"), torch.tensor(w, device="cuda"), ref, out)
    # sums of at most 3e5 FP64 terms of one sign: far below 1e-12
    assert np.abs(out.cpu().numpy() - want).max() <= 1e-12
    m.mbis_credible_levels(n, torch.tensor(theta, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda"),
                           ref, out)
    assert np.isnan(out.cpu().numpy()).all()
