"""The fixed-point FP64 likelihood against the oracle where its shape changes: part of a tile
and several tiles, less than one chunk of bins per warp up to clusters of sixteen CTAs, folded
and per-detector tables of one to four detectors, each marginalisation; data spanning many
binades, samples outside the model, and data that are not finite."""
import numpy as np
import pytest

import oracle
import workloads
from oracle.events import true_params
from gpu_common import m, torch  # noqa: F401

pytestmark = pytest.mark.gpu

SLOTS = [workloads.MC, workloads.Q, workloads.CHI1, workloads.CHI2, workloads.TC]
SKY = [workloads.RA, workloads.DEC, workloads.PSI, workloads.IOTA]
MARGS = [0, workloads.MARG_PHASE, workloads.MARG_PHASE | workloads.MARG_DISTANCE]


def build(n_bins, df, n_det, marg, masses, seed):
    rng = np.random.default_rng(seed)
    names = ["H1", "L1", "V1"]
    v, x, y = workloads.network(names)
    v = np.concatenate([v, [[4.0e6, 3.0e6, -4.0e6]]])[:n_det]
    x = np.concatenate([x, [[0.6, -0.8, 0.0]]])[:n_det]
    y = np.concatenate([y, [[0.0, 0.0, 1.0]]])[:n_det]
    f = 20.0 + df * np.arange(n_bins)
    psd = np.tile(oracle.psd_aligo(f), (n_det, 1))
    ev = oracle.OracleEvent(20.0, df, n_bins, psd, v, x, y, gmst=1.3, marg=marg)
    spec = workloads.EventSpec(masses[0], masses[1], dict(chi1=0.1, chi2=-0.05, ra=1.0, dec=0.5, psi=0.3, iota=0.4,
                                                          tc=0.01, phic=0.7), 1.3, 20.0, None, 1)
    th = true_params(spec, dl=1.0)
    rho = np.sqrt(max(oracle.optimal_snr2(ev, th), 1e-30))
    th[workloads.DL] = max(rho / 20.0, 20.0)
    ev.set_strain(oracle.make_strain(ev, th, seed, True))
    return ev, th, rng


def samples(ev, th, ids, n, rng):
    full = np.tile(th, (n, 1))
    full[:, workloads.MC] *= 1 + 1e-4 * rng.normal(size=n)
    full[:, workloads.Q] = 1 + np.abs(full[:, workloads.Q] - 1 + 0.05 * rng.normal(size=n))
    full[:, workloads.CHI1] += 0.02 * rng.normal(size=n)
    full[:, workloads.TC] += 1e-3 * rng.normal(size=n)
    if workloads.RA in ids:
        full[:, SKY] += 0.2 * rng.normal(size=(n, 4))
    if n > 20:  # heavier and lighter samples beside the rest: other cuts, other phase scales
        full[3, workloads.MC] *= 3.0
        full[4, workloads.MC] *= 0.4
        full[5, workloads.CHI1] = 1.2
        full[6, workloads.MC] = -1.0
        full[7, workloads.TC] = np.nan
    return full


def device(m, torch, ev, th, ids, marg, full):
    dets = m.make_detectors(ev.vertex, ev.xarm, ev.yarm)
    ctx = m.mbis_create(ev.strain[..., 0] + 1j * ev.strain[..., 1], ev.psd, dets, ev.s.f_lo, ev.s.df, th, gmst=1.3,
                        precision=m.FP64, marg=marg)
    try:
        P = len(ids)
        lo = np.array([{workloads.MC: 0.01, workloads.Q: 0.5, workloads.CHI1: -0.9, workloads.CHI2: -0.9,
                        workloads.TC: -1.0, workloads.DEC: -1.5, workloads.IOTA: 0.01}.get(s, 0.0) for s in ids])
        hi = np.array([{workloads.MC: 200.0, workloads.Q: 30.0, workloads.CHI1: 0.9, workloads.CHI2: 0.9,
                        workloads.TC: 1.0, workloads.DEC: 1.5, workloads.IOTA: 3.1}.get(s, 6.0) for s in ids])
        m.mbis_set_metric(ctx, np.array(ids, np.int32), th[ids], np.eye(P) * 1e-3, 1.0, lo, hi, 0)
        n = len(full)
        theta = torch.tensor(np.ascontiguousarray(full[:, ids].T), dtype=torch.float64, device="cuda")
        out = torch.empty(n, dtype=torch.float64, device="cuda")
        m.mbis_loglike(ctx, n, theta, out)
        return out.cpu().numpy()
    finally:
        m.mbis_destroy(ctx)


def check(got, want):
    assert np.array_equal(np.isfinite(got), np.isfinite(want))
    ok = np.isfinite(want)
    assert np.array_equal(got[~ok & ~np.isnan(want)], want[~ok & ~np.isnan(want)])
    # both sides round a phase of up to a few 10^3 turns at 2^-53: 10^-11 rad of |Z| up to 10^3
    assert np.all(np.abs(got[ok] - want[ok]) <= 1e-8 * np.maximum(1.0, np.abs(want[ok]) / 100.0))


def distance_rule(Z, H, dmin=10.0, dmax=1000.0):
    """The device's distance quadrature in numpy (48 points over +-12 widths of the peak, 8
    panels of 8 points on either side; 24 panels without a peak)."""
    from scipy.special import ive
    x48, w48 = np.polynomial.legendre.leggauss(48)
    x8, w8 = np.polynomial.legendre.leggauss(8)
    lo, hi = -np.log(dmax), -np.log(dmin)

    def rule(a, b, panels, x, w):
        h = 0.5 * (b - a) / panels
        s = (a + h * (2 * np.arange(panels)[:, None] + 1 + x)).ravel()
        return s, np.tile(h * w, panels)

    parts = [rule(lo, hi, 24, x8, w8)]
    if H > 0 and Z * Z > 14 * H:
        u = (Z + np.sqrt(Z * Z - 14 * H)) / (2 * H)
        sig, sc = 1 / np.sqrt(max(Z * u - 7, 1e-300)), np.log(u)
        wlo, whi = max(lo, sc - 12 * sig), min(hi, sc + 12 * sig)
        if wlo < whi:
            parts = [rule(wlo, whi, 1, x48, w48)]
            parts += [rule(lo, wlo, 8, x8, w8)] if wlo > lo else []
            parts += [rule(whi, hi, 8, x8, w8)] if whi < hi else []
    s, w = (np.concatenate(v) for v in zip(*parts))
    u = np.exp(s)
    g = np.log(3 / (dmax ** 3 - dmin ** 3)) - 3 * s + np.log(ive(0, Z * u)) + Z * u - 0.5 * H * u * u
    return g.max() + np.log((w * np.exp(g - g.max())).sum())


def expected(ev, full, marg):
    """The oracle's log L; with the distance marginalised, the device's quadrature of the
    oracle's overlap and norm (the two sides' rules differ where the range cuts the integrand
    off), which its plain log L at two distances and two phases gives."""
    want = oracle.loglike_batch(ev, full)
    if not marg & workloads.MARG_DISTANCE:
        return want
    ok = np.isfinite(want)
    plain, d = ev.with_marg(0), full[:, workloads.DL]
    z = []
    for phase in (0.0, np.pi / 2):
        p = full[ok].copy()
        p[:, workloads.PHIC] = phase
        l1 = oracle.loglike_batch(plain, p)
        p[:, workloads.DL] *= 2
        x = 4 * oracle.loglike_batch(plain, p) - l1
        z.append((x * d[ok], 2 * (x - l1) * d[ok] ** 2))
    want[ok] = [distance_rule(np.hypot(a, b), h) for (a, b, h) in zip(z[0][0], z[1][0], z[0][1])]
    return want


@pytest.mark.parametrize("n_bins,n", [(7, 1), (255, 31), (513, 33), (2049, 95), (9000, 40), (40000, 33)])
@pytest.mark.parametrize("marg", MARGS)
def test_folded_against_the_oracle(m, torch, n_bins, n, marg):  # noqa: F811
    ev, th, rng = build(n_bins, 0.25 if n_bins < 3000 else 1 / 64, 2, marg, (30.0, 25.0) if n_bins < 3000 else (1.5, 1.3),
                        n_bins)
    full = samples(ev, th, SLOTS, n, rng)
    check(device(m, torch, ev, th, SLOTS, marg, full), expected(ev, full, marg))


@pytest.mark.parametrize("n_det", [1, 2, 3, 4])
@pytest.mark.parametrize("marg", MARGS)
def test_per_detector_against_the_oracle(m, torch, n_det, marg):  # noqa: F811
    ev, th, rng = build(3001, 0.125, n_det, marg, (12.0, 9.0), 10 + n_det)
    full = samples(ev, th, SLOTS + SKY, 70, rng)
    check(device(m, torch, ev, th, SLOTS + SKY, marg, full), expected(ev, full, marg))


def test_wide_range_of_data_and_not_finite_data(m, torch):  # noqa: F811
    ev, th, rng = build(2000, 0.25, 2, workloads.MARG_PHASE, (30.0, 25.0), 3)
    full = samples(ev, th, SLOTS, 40, rng)
    ev.strain[:, 100] *= 1e12       # one loud line among the other 31 bins of its chunk
    ev.strain[:, 101] *= 1e-40
    ev.strain[:, 64:96] = 0.0       # an empty chunk
    want, got = oracle.loglike_batch(ev, full), device(m, torch, ev, th, SLOTS, workloads.MARG_PHASE, full)
    ok = np.isfinite(want)
    # |Z| is the loud bin's: relative rounding
    assert np.all(np.abs(got[ok] - want[ok]) <= 1e-11 * np.abs(want[ok]))
    ev.strain[0, 10] = np.nan
    got = device(m, torch, ev, th, SLOTS, workloads.MARG_PHASE, full)
    assert np.all(np.isnan(got[np.isfinite(want)]))
