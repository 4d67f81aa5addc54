"""The one-launch weight reduction where its shape changes: fewer samples than one CTA, one
sample per thread, several kept in registers, and more than the registers keep (the inputs
are then read twice); whole CTAs without a finite weight; weights written over an input."""
import numpy as np
import pytest

import oracle
from gpu_common import m, torch  # noqa: F401
from test_zz_no_alloc import TOL, _context

pytestmark = pytest.mark.gpu

GRID = 608 * 256  # threads of the largest launch


@pytest.mark.parametrize("n", [1, 255, 257, GRID, GRID + 1, 8 * GRID, 8 * GRID + 1, 3_000_017])
@pytest.mark.parametrize("alias", [False, True])
def test_reduce_against_the_oracle_at_the_launch_edges(m, torch, n, alias):  # noqa: F811
    rng = np.random.default_rng(n)
    ll, lp, lq = rng.normal(40.0, 6.0, n), rng.normal(-2.0, 0.5, n), rng.normal(-1.0, 1.0, n)
    if n > 1000:
        lp[:700] = -np.inf           # CTAs 0 and 1 hold no finite weight at the small sizes
        ll[n // 2:n // 2 + 300] -= 800.0  # underflows against the maximum
    want = oracle.reduce(ll, lp, lq, want_weights=True)
    ctx = _context(m)
    try:
        d = [torch.tensor(a, dtype=torch.float64, device="cuda") for a in (ll, lp, lq)]
        w = d[0] if alias else torch.empty(n, dtype=torch.float64, device="cuda")
        got = m.mbis_reduce(ctx, n, *d, w)
        assert got["n"] == n and got["max_logw"] == want["max_logw"]
        assert abs(got["ess"] / want["ess"] - 1) < TOL
        assert abs(got["log_z"] - want["log_z"]) < TOL * max(1.0, abs(want["log_z"]))
        np.testing.assert_allclose(w.cpu().numpy(), want["weights"], rtol=TOL, atol=1e-300)
    finally:
        m.mbis_destroy(ctx)
