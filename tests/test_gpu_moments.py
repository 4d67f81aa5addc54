"""Weighted moments for every slot count (one instantiation each), at sample counts around a
warp, a CTA and the largest grid, with zero, negative and NaN weights and periodic slots whose
samples lie on both sides of their period."""
import numpy as np
import pytest

import oracle
from gpu_common import m, torch  # noqa: F401

pytestmark = pytest.mark.gpu

IDS = [4, 0, 10, 1, 6, 2, 3, 5, 7, 8, 9]  # RA, phi_c and psi (periodic) among the first five


def moments_context(m, P, mean, chol):
    dets = m.make_detectors([[0.0, 0.0, 6.4e6]], [[1.0, 0.0, 0.0]], [[0.0, 1.0, 0.0]])
    ctx = m.mbis_create(np.zeros((1, 8), dtype=np.complex128), np.ones((1, 8)), dets, 20.0, 1.0,
                        [1.2, 1.1, 0, 0, 0, 0, 0, 0, 100.0, 0, 0], precision=m.FP64, marg=0)
    m.mbis_set_metric(ctx, IDS[:P], mean, chol, 1.0, np.full(P, 0.01), np.full(P, 1.5))
    return ctx


@pytest.mark.parametrize("P", range(1, 12))
@pytest.mark.parametrize("n", [1, 31, 257, 152 * 256 + 1, 100_003])
def test_moments_for_every_slot_count(m, torch, P, n):  # noqa: F811
    rng = np.random.default_rng(1000 * P + n)
    mean = rng.uniform(0.2, 1.0, P)
    theta = mean[:, None] + 0.4 * rng.normal(size=(P, n))
    for p, s in enumerate(IDS[:P]):
        if s in (4, 6, 10):  # wrapped into the period, so that some lie a period away
            theta[p] = np.mod(theta[p] + 0.3 * rng.normal(size=n) - 0.5, np.pi if s == 6 else 2 * np.pi)
    w = rng.exponential(size=n)
    if n > 30:
        w[1::7], w[2::11], w[3::13] = 0.0, -1.0, np.nan
    ctx = moments_context(m, P, mean, np.eye(P) * 0.1)
    try:
        got_m, got_c = m.mbis_weighted_moments(ctx, n, torch.tensor(theta, device="cuda"),
                                               torch.tensor(w, device="cuda"))
    finally:
        m.mbis_destroy(ctx)
    use = w > 0
    want_m, want_c = oracle.weighted_moments(IDS[:P], np.ascontiguousarray(theta[:, use]), w[use], mean)
    # the covariance is E[dd'] - E[d] E[d]' of the offsets d from the proposal mean; by the
    # standard bound on a sum of n rounded products (Higham, Accuracy and Stability of Numerical
    # Algorithms, ch. 3) each of the two sides is within (n + a few tens) u of the second moments
    gamma = 2 * (n + 64) * 2.0 ** -53
    off = want_m - mean
    for p, s in enumerate(IDS[:P]):
        if s in (4, 6, 10):
            off[p] = (off[p] + np.pi / 2) % np.pi - np.pi / 2 if s == 6 else (off[p] + np.pi) % (2 * np.pi) - np.pi
    rms = np.sqrt(np.diag(want_c) + off ** 2)
    assert np.all(np.abs(got_m - want_m) <= 2 * gamma * rms + 4 * 2.0 ** -53 * np.abs(want_m))
    assert np.all(np.abs(got_c - want_c) <= 2 * gamma * np.outer(rms, rms))
