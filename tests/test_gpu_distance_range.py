"""The distance marginal of sources that lie outside the distance prior: the integrand then has
its peak more than twelve widths beyond an end of [dmin, dmax] and the rule runs over the whole
range.  Events nearer than dmin, farther than dmax, in between, and too faint for a peak; through
the folded kernel (whole tiles and split over the bins' parts), a batch step, relative binning
with one bin per grid point, and the FP64 kernel, each against the rule in numpy on the oracle's
overlap and norm (the mixed kernels take half as many panels beside the peak's window)."""
import numpy as np
import pytest

import oracle
import workloads
from gpu_common import m, torch, logl_bound  # noqa: F401
from test_gpu_fp64 import SLOTS, build, samples

pytestmark = pytest.mark.gpu

MARG = workloads.MARG_PHASE | workloads.MARG_DISTANCE
DMIN, DMAX = 10.0, 1000.0
# distance (Mpc) and signal-to-noise ratio of the injection: the peak's width in ln d is 1 / 20 at
# a ratio of 20, so that 3000 and 4 Mpc lie 22 and 18 widths beyond the range's ends
SOURCES = {"far": (3000.0, 20.0), "near": (4.0, 20.0), "inside": (150.0, 20.0), "no peak": (300.0, 1.0)}


def event(n_bins, source):
    dl, snr = SOURCES[source]
    ev, th, rng = build(n_bins, 0.25 if n_bins < 3000 else 1 / 64, 2, MARG, (30.0, 25.0) if n_bins < 3000 else (1.5, 1.3),
                        7 + n_bins)
    th[workloads.DL] = dl
    scale = oracle.optimal_snr2(ev, th) / snr ** 2
    ev = oracle.OracleEvent(ev.s.f_lo, ev.s.df, n_bins, ev.psd * scale, ev.vertex, ev.xarm, ev.yarm, gmst=1.3, marg=MARG,
                            dmin=DMIN, dmax=DMAX)
    ev.set_strain(oracle.make_strain(ev, th, 5, False))
    return ev, th, rng


def context(m, ev, th, precision):
    dets = m.make_detectors(ev.vertex, ev.xarm, ev.yarm)
    ctx = m.mbis_create(ev.strain[..., 0] + 1j * ev.strain[..., 1], ev.psd, dets, ev.s.f_lo, ev.s.df, th, gmst=1.3,
                        precision=precision, marg=MARG, dmin=DMIN, dmax=DMAX)
    width = np.array([1e-5 * th[workloads.MC], 0.02, 0.01, 0.01, 1e-4])
    mean = th[SLOTS].copy()
    mean[1] += 0.2
    m.mbis_set_metric(ctx, np.array(SLOTS, np.int32), mean, np.diag(width), 1.0, mean - 5 * width, mean + 5 * width, 0)
    return ctx


def rule(Z, H, side_panels):
    """48 points over +-12 widths of the peak and side_panels panels of 8 on either side of them; 24
    panels over the whole range without a peak in it."""
    from scipy.special import ive
    x48, w48 = np.polynomial.legendre.leggauss(48)
    x8, w8 = np.polynomial.legendre.leggauss(8)
    lo, hi = -np.log(DMAX), -np.log(DMIN)

    def composite(a, b, panels, x, w):
        h = 0.5 * (b - a) / panels
        return (a + h * (2 * np.arange(panels)[:, None] + 1 + x)).ravel(), np.tile(h * w, panels)

    parts = [composite(lo, hi, 24, x8, w8)]
    if H > 0 and Z * Z > 14 * H:
        u = (Z + np.sqrt(Z * Z - 14 * H)) / (2 * H)
        sig, sc = 1 / np.sqrt(Z * u - 7), np.log(u)
        wlo, whi = max(lo, sc - 12 * sig), min(hi, sc + 12 * sig)
        if wlo < whi:
            parts = [composite(wlo, whi, 1, x48, w48)]
            parts += [composite(lo, wlo, side_panels, x8, w8)] if wlo > lo else []
            parts += [composite(whi, hi, side_panels, x8, w8)] if whi < hi else []
    s, w = (np.concatenate(v) for v in zip(*parts))
    u = np.exp(s)
    g = np.log(3 / (DMAX ** 3 - DMIN ** 3)) - 3 * s + np.log(ive(0, Z * u)) + Z * u - 0.5 * H * u * u
    return g.max() + np.log((w * np.exp(g - g.max())).sum())


def expected(ev, full, side_panels):
    """The rule on the oracle's overlap and norm, which its plain log L at two distances and two
    phases gives; not finite outside the model."""
    want = oracle.loglike_batch(ev, full)
    ok = np.isfinite(want)
    plain, d = ev.with_marg(0), full[ok, workloads.DL]
    z = []
    for phase in (0.0, np.pi / 2):
        p = full[ok].copy()
        p[:, workloads.PHIC] = phase
        l1 = oracle.loglike_batch(plain, p)
        p[:, workloads.DL] *= 2
        x = 4 * oracle.loglike_batch(plain, p) - l1
        z.append((x * d, 2 * (x - l1) * d ** 2))
    want[ok] = [rule(np.hypot(a, b), h, side_panels) for a, b, h in zip(z[0][0], z[1][0], z[0][1])]
    return want


def check(got, want):
    assert np.array_equal(np.isfinite(got), np.isfinite(want)), (got[:8], want[:8])
    ok = np.isfinite(want)
    d = np.abs(got[ok] - want[ok])
    assert np.all(d <= logl_bound(want[ok])), d.max()


@pytest.mark.parametrize("source", list(SOURCES))
@pytest.mark.parametrize("n_bins", [2049, 9000])  # whole tiles; two parts of 8192 bins
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_likelihood_outside_the_distance_range(m, torch, n_bins, source, precision):  # noqa: F811
    ev, th, rng = event(n_bins, source)
    full = samples(ev, th, SLOTS, 70, rng)
    ctx = context(m, ev, th, m.MIXED if precision == "mixed" else m.FP64)
    try:
        theta = torch.tensor(np.ascontiguousarray(full[:, SLOTS].T), dtype=torch.float64, device="cuda")
        out = torch.empty(len(full), dtype=torch.float64, device="cuda")
        m.mbis_loglike(ctx, len(full), theta, out)
        want = expected(ev, full, 4 if precision == "mixed" else 8)
        check(out.cpu().numpy(), want)
        if precision == "mixed":
            m.mbis_rb_setup(ctx, th, np.arange(n_bins + 1, dtype=np.int32))
            m.mbis_rb_loglike(ctx, len(full), theta, out)
            # but for the two of another mass: their phases' FP32 differences from the fiducial's
            # are thousands of turns
            near = np.delete(np.arange(len(full)), [3, 4])
            check(out.cpu().numpy()[near], want[near])
    finally:
        m.mbis_destroy(ctx)


def test_batch_of_sources_outside_the_distance_range(m, torch):  # noqa: F811
    evs = [event(2049, s) for s in SOURCES]
    ctxs = [context(m, ev, th, m.MIXED) for ev, th, _ in evs]
    n = 100
    b = m.mbis_batch_create(ctxs, [n] * len(ctxs), [11 + i for i in range(len(ctxs))])
    try:
        sums = m.mbis_batch_step(b, 0, len(ctxs))
        for i, (ev, th, _) in enumerate(evs):
            theta, ll = m.mbis_batch_copy_out(b, i, len(SLOTS), n)
            check(ll, expected(ev, oracle.full_params(SLOTS, theta, th), 4))
            assert np.isfinite(sums[i]["log_z"]) and sums[i]["ess"] > 0.999
    finally:
        m.mbis_batch_destroy(b)
        for c in ctxs:
            m.mbis_destroy(c)
