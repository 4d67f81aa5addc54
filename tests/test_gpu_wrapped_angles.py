"""Periodic slots drawn a few ulps, or far less, on either side of their period's ends stay inside
[0, period) in both arithmetics."""
import numpy as np
import pytest

from gpu_common import m, torch  # noqa: F401

pytestmark = pytest.mark.gpu

RA, PSI, PHIC = 4, 6, 10
PERIOD = {RA: 2 * np.pi, PHIC: 2 * np.pi, PSI: np.pi}


def draws(m, torch, slot, mean, width, precision, lo=0.0, hi=1.0, n=4096):  # noqa: F811
    dets = m.make_detectors([[0.0, 0.0, 6.4e6]], [[1.0, 0.0, 0.0]], [[0.0, 1.0, 0.0]])
    fixed = [1.3, 1.6, 0.0, 0.0, 0.5, 0.3, 0.2, 0.9, 300.0, 0.0, 0.1]
    ctx = m.mbis_create(np.ones((1, 64), dtype=np.complex128), np.ones((1, 64)), dets, 20.0, 1.0, fixed,
                        precision=m.FP64 if precision == "fp64" else m.MIXED,
                        marg=m.MARG_TIME if precision == "mixed" else 0)
    try:
        m.mbis_set_metric(ctx, np.array([slot], np.int32), [mean], [[width]], 1.0, [lo], [hi], 0)
        th = torch.empty((1, n), dtype=torch.float64, device="cuda")
        lq, lp = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
        m.mbis_draw(ctx, 31, 0, n, th, lq, lp)
        return th[0].cpu().numpy(), lp.cpu().numpy()
    finally:
        m.mbis_destroy(ctx)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("slot", [RA, PSI, PHIC])
@pytest.mark.parametrize("turns,width", [(0, 1e-50), (0, 1e-20), (0, 2e-16), (0, 1e-15), (1, 1e-15), (-1, 1e-15), (3, 1e-14),
                                         (-3, 1e-14), (1, 1e-9)])
def test_wrapped_angles_stay_in_their_period(m, torch, slot, turns, width, precision):  # noqa: F811
    T = PERIOD[slot]
    got, lp = draws(m, torch, slot, turns * T, width, precision)
    assert got.min() >= 0.0 and got.max() < T, (got.min(), got.max() - T)
    # within the draws' reach (4096 normals: 5 of them) and an ulp of the period of one of its ends
    assert np.all(np.minimum(got, T - got) <= 5 * width + 4 * 2.0 ** -52 * max(1, abs(turns)) * T)
    assert np.allclose(lp, -np.log(T), rtol=1e-15, atol=0)
