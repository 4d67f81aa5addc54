"""Draws of every slot count (one instantiation each) in both arithmetics against the oracle:
fixed-point normals (FP64 contexts) and library normals (mixed contexts), with periodic,
trigonometric, distance and mass priors among the slots, at sample counts around a CTA, a
Cholesky factor spanning many binades, and counters beyond 32 bits."""
import numpy as np
import pytest

import oracle
from gpu_common import m, torch  # noqa: F401

pytestmark = pytest.mark.gpu

IDS = [0, 1, 4, 5, 6, 7, 8, 9, 10, 2, 3]
MEAN = dict(zip(range(11), [1.3, 1.6, 0.1, -0.1, 3.0, 0.4, 1.5, 1.2, 300.0, 0.0, 3.1]))
WIDTH = dict(zip(range(11), [1e-4, 0.1, 0.02, 0.03, 2.0, 0.5, 1.0, 0.6, 80.0, 1e-3, 3.0]))
LO = dict(zip(range(11), [1.0, 1.0, -0.9, -0.9, 0.0, -1.5, 0.0, 0.01, 10.0, -1.0, 0.0]))
HI = dict(zip(range(11), [2.0, 4.0, 0.9, 0.9, 6.2, 1.5, 3.1, 3.1, 1000.0, 1.0, 6.2]))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("P", range(1, 12))
def test_draws_of_every_slot_count(m, torch, P, precision):  # noqa: F811
    rng = np.random.default_rng(P)
    ids = np.array(IDS[:P], np.int32)
    dets = m.make_detectors([[0.0, 0.0, 6.4e6]], [[1.0, 0.0, 0.0]], [[0.0, 1.0, 0.0]])
    ctx = m.mbis_create(np.ones((1, 512), dtype=np.complex128), np.ones((1, 512)), dets, 20.0, 1.0,
                        [MEAN[s] for s in range(11)], precision=m.FP64 if precision == "fp64" else m.MIXED,
                        marg=m.MARG_TIME if precision == "mixed" else 0)
    mean = np.array([MEAN[s] for s in ids])
    chol = np.diag([WIDTH[s] for s in ids]) @ (np.eye(P) + np.tril(rng.normal(0, 0.3, (P, P)), -1))
    lo, hi = np.array([LO[s] for s in ids]), np.array([HI[s] for s in ids])
    flags = m.PRIOR_M1M2 if P >= 2 else 0
    try:
        m.mbis_set_metric(ctx, ids, mean, chol, 1.25, lo, hi, flags)
        for n, ctr0 in ((1, 0), (127, 5), (129, 2 ** 32 - 40), (5000, 2 ** 40)):
            th = torch.empty((P, n), dtype=torch.float64, device="cuda")
            lq, lp = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
            m.mbis_draw(ctx, 77, ctr0, n, th, lq, lp)
            want, want_q = oracle.draw(77, ctr0, n, ids, mean, chol, 1.25)
            got = th.cpu().numpy()
            for p, s in enumerate(ids):
                d = np.abs(got[p] - want[p])
                if s in (4, 6, 10):  # a point at a period's end may round to either
                    d = np.minimum(d, np.abs(d - (np.pi if s == 6 else 2 * np.pi)))
                assert np.all(d <= 1e-12 * max(1.0, abs(MEAN[int(s)]))), (P, s, d.max())
            np.testing.assert_allclose(lq.cpu().numpy(), want_q, rtol=1e-12, atol=1e-12)
            want_p = oracle.log_prior(ids, lo, hi, flags, got)
            got_p = lp.cpu().numpy()
            assert np.array_equal(np.isfinite(got_p), np.isfinite(want_p))
            ok = np.isfinite(want_p)
            # log cos and log sin near their zeros carry the angle's rounding: 1e-15 / 1e-3
            np.testing.assert_allclose(got_p[ok], want_p[ok], rtol=1e-12, atol=1e-12)
    finally:
        m.mbis_destroy(ctx)
