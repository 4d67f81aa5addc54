"""The normalised weights to their last bits: each is one exponential, one reciprocal and one
product, whichever CTA its sample belongs to, so that samples of one log weight get one weight."""
import numpy as np
import pytest

from gpu_common import m, torch  # noqa: F401
from test_zz_no_alloc import _context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5000, 608 * 256 + 77, 2_000_003])
def test_weights_to_their_last_bits(m, torch, n):  # noqa: F811
    rng = np.random.default_rng(n)
    # eighths: the sums and the differences from the largest are exact, and values repeat
    ll, lp, lq = (np.round(rng.normal(mu, sd, n) * 8) / 8 for mu, sd in ((40.0, 6.0), (-2.0, 0.5), (-1.0, 1.0)))
    ctx = _context(m)
    try:
        w = torch.empty(n, dtype=torch.float64, device="cuda")
        s = m.mbis_reduce(ctx, n, *(torch.tensor(a, device="cuda") for a in (ll, lp, lq)), w)
    finally:
        m.mbis_destroy(ctx)
    w, lw = w.cpu().numpy(), ll + lp - lq
    want = np.exp((lw - lw.max()).astype(np.longdouble)) / np.longdouble(s["s1"])
    # 0.8 ulp of the exponential, half an ulp of the reciprocal and of the product; an ulp is at
    # most 2^-52 of its number
    err = np.abs(w / want - 1).max()
    assert err <= 1.8 * 2.0 ** -52, err * 2.0 ** 52
    order = np.argsort(lw, kind="stable")
    same = np.diff(lw[order]) == 0
    assert np.array_equal(w[order][1:][same], w[order][:-1][same])
