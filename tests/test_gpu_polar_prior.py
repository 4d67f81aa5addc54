"""The log prior of a drawn declination or inclination keeps its relative accuracy up to the poles,
in both arithmetics."""
import numpy as np
import pytest

from gpu_common import m, torch  # noqa: F401
from test_gpu_wrapped_angles import draws

pytestmark = pytest.mark.gpu

DEC, IOTA = 5, 7


@pytest.mark.parametrize("off", [0.3, 0.13, 0.121, 0.119, 0.05, 1e-2, 1e-3, 1e-4, 1e-6, 1e-8, 1e-12, 1e-100])
@pytest.mark.parametrize("slot,pole", [(IOTA, 0.0), (IOTA, np.pi), (DEC, np.pi / 2), (DEC, -np.pi / 2)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_log_prior_near_the_poles(m, torch, slot, pole, off, precision):  # noqa: F811
    lo, hi = (0.0, np.pi) if slot == IOTA else (-np.pi / 2, np.pi / 2)
    got, lp = draws(m, torch, slot, pole - np.copysign(off, pole - 0.1), 0.01 * off, precision, lo, hi)
    inside = (got >= lo) & (got <= hi)
    assert np.array_equal(np.isfinite(lp), inside) and inside.any()
    x = got[inside].astype(np.longdouble)
    want = np.log(np.sin(x) if slot == IOTA else np.cos(x)) - np.log(np.longdouble(2))
    # a sine and its logarithm within an ulp each, the prior's constant and the sum rounded once
    assert np.all(np.abs(lp[inside] - want) <= 2.0 ** -52 * (2 + 2 * np.abs(want)))


def test_log_prior_at_the_face_on_pole(m, torch):  # noqa: F811
    got, lp = draws(m, torch, IOTA, 0.0, 5e-324, "fp64", 0.0, np.pi, 64)
    assert np.all(np.isneginf(lp[got == 0.0])) and (got == 0.0).any()
