"""Performance cases of the library: what its users run, at the sizes they run it.

A user of the library holds events (strain, PSD, detectors, a Gaussian proposal) and asks for
draws, log likelihoods, importance weights and posterior summaries.  Each case is one such
call or one short sequence of calls through the package's public entry points; `kind` names
the sequence and the other keys its sizes.  Inputs (events and samples) are made here from
the seed with numpy and torch alone, so that `exact` states the same quantities in 64 bits
without the library.
"""
import math

import numpy as np
import torch

import paper_2410_05190_gb300 as mbis

MC, Q, CHI1, CHI2, RA, DEC, PSI, IOTA, DL, TC, PHIC = range(11)
MTSUN = 4.925490947641267e-6                       # G Msun / c^3, s
CLIGHT = 299792458.0
MPC_S = 3.0856775814913673e22 / CLIGHT             # 1 Mpc / c, s
DMIN, DMAX = 10.0, 1000.0                          # distance prior, Mpc
N_SHIFT, DT_SHIFT = 128, 1e-4                      # time marginalisation
INV_2_32 = 2.0 ** -32

# LIGO Hanford, LIGO Livingston, Virgo: vertex (m) and unit arms (Anderson et al. 2001)
SITES = [
    ((-2161414.92636, -3834695.17889, 4600350.22664), (-0.22389266154, 0.79983062746, 0.55690487831),
     (-0.91397818574, 0.02609403989, -0.40492342125)),
    ((-74276.0447238, -5496283.71971, 3224257.01744), (-0.95457412153, -0.14158077340, -0.26218911324),
     (0.29774156894, -0.48791033647, -0.82054461286)),
    ((4546374.099, 842989.6976, 4378576.963), (-0.70045821479, 0.20848948619, 0.68256166277),
     (-0.05379255368, -0.96908180549, 0.24080451708)),
]

# The source families: masses, spins, SNR, band, sampled slots, marginalisation, proposal width.
#   heavy  two heavy black holes, intrinsic parameters only, phase marginalised
#   bns    neutron stars: long signals, (Mc, q, chi1, chi2, t_c), phase and distance marginalised
#   bbhx   black holes, intrinsic parameters and t_c, phase and distance marginalised
#   bbh    black holes with every parameter sampled, time marginalised over 128 shifts
FAMILY = {
    "heavy": dict(m=(20.0, 40.0), chi=0.5, snr=(10.0, 30.0), f_hi=512.0, ids=[MC, Q, CHI1, CHI2],
                  marg=mbis.MARG_PHASE, scale=1.5, flags=0),
    "bns": dict(m=(1.1, 2.0), chi=0.05, snr=(10.0, 30.0), f_hi=1024.0, ids=[MC, Q, CHI1, CHI2, TC],
                marg=mbis.MARG_PHASE | mbis.MARG_DISTANCE, scale=1.5, flags=mbis.PRIOR_M1M2),
    "bbhx": dict(m=(10.0, 80.0), chi=0.8, snr=(10.0, 40.0), f_hi=1024.0, ids=[MC, Q, CHI1, CHI2, TC],
                 marg=mbis.MARG_PHASE | mbis.MARG_DISTANCE, scale=1.5, flags=mbis.PRIOR_M1M2),
    "bbh": dict(m=(10.0, 80.0), chi=0.8, snr=(10.0, 40.0), f_hi=1024.0, ids=list(range(11)),
                marg=mbis.MARG_TIME, scale=1.5, flags=mbis.PRIOR_M1M2),
}
F_LO = 20.0
# The two-parameter demonstration space of the tiled proposal
SPACE = dict(x_lo=20.0, x_hi=28.0, mc_period=4.0, mc_base=24.0, q_lo=1.0 / 6.0, q_hi=6.0)
TILE_F_HI, TILE_DF = 128.0, 0.25


def listed():
    return [
        # The smallest call: one event of 1969 bins, 4096 proposal points, double precision
        # throughout; a full importance-sampling pass (draw, likelihood, weights), where
        # launches and latency count.
        dict(name="pass_fp64_tiny", kind="pass", family="heavy", precision="fp64", df=0.25, det=2, n=4096, c128=True),
        # The double-precision check of a neutron-star event on its full grid.
        dict(name="loglike_fp64_bns", kind="loglike", family="bns", precision="fp64", df=1 / 128, det=2, n=4096,
             c128=False),
        # The population workload: 2^20 points on 128,513 bins, mixed precision.  The largest.
        dict(name="loglike_bns_population", kind="loglike", family="bns", precision="mixed", df=1 / 128, det=2,
             n=1 << 20, c128=False),
        # One batch of the ESS-target loop on the same grid.
        dict(name="loglike_bns_batch", kind="loglike", family="bns", precision="mixed", df=1 / 128, det=2, n=1 << 16,
             c128=False),
        # Short signals with fixed sky (the black-hole P-P population): 8033 bins, three
        # detectors, one refit batch; the per-sample work weighs against few bins.
        dict(name="loglike_bbh_intrinsic", kind="loglike", family="bbhx", precision="mixed", df=1 / 8, det=3, n=1 << 16,
             c128=False),
        # Eleven sampled parameters, time marginalised on the tensor cores, a population launch.
        dict(name="loglike_bbh_time", kind="loglike", family="bbh", precision="mixed", df=1 / 8, det=3, n=1 << 18,
             c128=False),
        # The same likelihood on a small ragged set of points (a re-evaluation of the heaviest
        # samples): fewer tiles than the GPU has multiprocessors.
        dict(name="loglike_bbh_time_small", kind="loglike", family="bbh", precision="mixed", df=1 / 8, det=3, n=3001,
             c128=False),
        # Events of uneven grids, detector counts and sample counts in one batched step.
        dict(name="batch_uneven", kind="batch", events=8, log2_n=14),
        # A whole run to a target ESS with proposal refits, on the relative-binning likelihood.
        dict(name="ess_relative_binning", kind="ess", family="bns", df=1 / 128, det=2, batch=1 << 16),
        # Proposal draws with every parameter sampled.
        dict(name="draw_all_parameters", kind="draw", family="bbh", n=1 << 18),
        # What follows the likelihoods of an event: weights and evidence, the weighted mean and
        # covariance of a refit, the credible levels of a P-P test.
        dict(name="posterior_stage", kind="stage", p=5, n=1 << 18),
        # Tile assignment of a pool of prior points to a template bank.
        dict(name="tile_assignment", kind="tiles", n=1 << 20),
    ]


def _log_int(rng, lo, hi):
    """An odd-or-even whole number, uniform in its logarithm over [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["loglike", "loglike", "loglike", "loglike", "pass", "batch", "ess", "draw", "stage", "tiles"])
    if kind in ("loglike", "pass"):
        family = rng.choice(list(FAMILY))
        precision = rng.choice(["mixed", "mixed", "mixed", "fp64"]) if kind == "loglike" else "fp64"
        df = math.exp(rng.uniform(math.log(1 / 128), math.log(1 / 4)))  # bin counts of every parity
        k = _n_bins(family, df)
        # sample-bins of a pass: at most those of the population launch (mixed), or what double
        # precision does in a few tens of milliseconds
        cost = (6e10 if family != "bbh" else 4e9) if precision == "mixed" else (6e8 if family != "bbh" else 4e7)
        return dict(kind=kind, family=family, precision=precision, df=df, det=rng.choice([2, 3]),
                    n=_log_int(rng, 1000, max(1001, min(1 << 20, cost / k))), c128=rng.random() < 0.3)
    if kind == "batch":
        return dict(kind=kind, events=rng.randint(2, 12), log2_n=rng.choice([12, 13, 14]))
    if kind == "ess":
        return dict(kind=kind, family="bns", df=rng.choice([1 / 128, 1 / 64, 1 / 32]), det=rng.choice([2, 3]),
                    batch=_log_int(rng, 1 << 13, 1 << 17))
    if kind == "draw":
        return dict(kind=kind, family=rng.choice(list(FAMILY)), n=_log_int(rng, 1000, 1 << 20))
    if kind == "stage":
        return dict(kind=kind, p=rng.choice([2, 4, 5, 11]), n=_log_int(rng, 1000, 1 << 21))
    return dict(kind="tiles", n=_log_int(rng, 5000, 1 << 21))


# ---------------------------------------------------------------------------- the model
# TaylorF2 with aligned spins to 3.5PN, f^-7/6 amplitude, zero at and above the ISCO, in plain
# torch; the event's data, its metric and the 64-bit answers all come from here.

def _n_bins(family, df):
    return int((FAMILY[family]["f_hi"] - F_LO) / df + 1e-9) + 1


def _psd(f):
    x = f / 215.0
    x2 = x * x
    return 1e-49 * (x ** -4.14 - 5.0 / x2 + 111.0 * (1.0 - x2 + 0.5 * x2 * x2) / (1.0 + 0.5 * x2))


def _mass_seconds(mc, q):
    return mc * MTSUN * (1.0 + q) ** 1.2 * q ** -0.6


def _isco(mc, q):
    return 1.0 / (6.0 ** 1.5 * math.pi * _mass_seconds(mc, q))


def _basis(f):
    c, lf = f ** (1.0 / 3.0), torch.log(f)
    return torch.stack([1.0 / (f * c * c), 1.0 / f, 1.0 / (c * c), 1.0 / c, lf, c, c * lf, c * c, f,
                        torch.ones_like(f)])


def _coeffs(mc, q, chi1, chi2, tc, phic):
    """[10][n]: the phase in turns is their sum with _basis."""
    pi = math.pi
    eta, dm = q / (1.0 + q) ** 2, (q - 1.0) / (q + 1.0)
    xs, xa = 0.5 * (chi1 + chi2), 0.5 * (chi1 - chi2)
    e2, e3 = eta * eta, eta ** 3
    p2 = 3715 / 756 + 55 / 9 * eta
    p3 = -16 * pi + 113 / 3 * dm * xa + (113 / 3 - 76 / 3 * eta) * xs
    p4 = (15293365 / 508032 + 27145 / 504 * eta + 3085 / 72 * e2 + (-405 / 8 + 200 * eta) * xa * xa
          - 405 / 4 * dm * xa * xs + (-405 / 8 + 5 / 2 * eta) * xs * xs)
    c5 = (pi * (38645 / 756 - 65 / 9 * eta) + dm * (-732985 / 2268 - 140 / 9 * eta) * xa
          + (-732985 / 2268 + 24260 / 81 * eta + 340 / 9 * e2) * xs)
    a6 = (11583231236531 / 4694215680 - 640 / 3 * pi ** 2 - 6848 / 21 * (0.5772156649015329 + math.log(4.0))
          + (-15737765635 / 3048192 + 2255 / 12 * pi ** 2) * eta + 76055 / 1728 * e2 - 127825 / 1296 * e3
          + pi * (2270 / 3 * dm * xa + (2270 / 3 - 520 * eta) * xs)
          + (75515 / 144 - 8225 / 18 * eta) * dm * xa * xs
          + (75515 / 288 - 263245 / 252 * eta - 480 * e2) * xa * xa
          + (75515 / 288 - 232415 / 504 * eta + 1255 / 9 * e2) * xs * xs)
    p7 = (pi * (77096675 / 254016 + 378515 / 1512 * eta - 74045 / 756 * e2)
          + (-25150083775 / 3048192 + 10566655595 / 762048 * eta - 1042165 / 3024 * e2 + 5345 / 36 * e3) * xs
          + dm * (-25150083775 / 3048192 + 26804935 / 6048 * eta - 1985 / 48 * e2) * xa)
    a = pi * _mass_seconds(mc, q)
    la, a13 = torch.log(a), a ** (1.0 / 3.0)
    pre = 3.0 / (128.0 * eta) / (2.0 * pi)
    return torch.stack([pre / (a * a13 * a13), pre * p2 / a, pre * p3 / (a13 * a13), pre * p4 / a13, pre * c5,
                        pre * a13 * (a6 - 6848 / 63 * la), -pre * a13 * (6848 / 63), pre * p7 * a13 * a13, tc,
                        -phic / (2 * pi) - 0.125 + pre * c5 * (1.0 + la)])


def _amplitude(mc, dl):
    return math.sqrt(5.0 / 24.0) * math.pi ** (-2.0 / 3.0) * (mc * MTSUN) ** (5.0 / 6.0) / (dl * MPC_S)


def _responses(ra, dec, psi, iota, gmst, n_det):
    """Per detector (Re P, Im P, delay): h = A f^-7/6 P e^(-i (Psi + 2 pi f delay))."""
    ph = ra - gmst
    sp, cp, sd, cd, ss, cs = ph.sin(), ph.cos(), dec.sin(), dec.cos(), psi.sin(), psi.cos()
    X = (sp * cs - ss * cp * sd, -cp * cs - ss * sp * sd, ss * cd)
    Y = (-sp * ss - cs * cp * sd, cp * ss - cs * sp * sd, cs * cd)
    ci = iota.cos()
    out = []
    for r, x, y in SITES[:n_det]:
        xX, xY = sum(u * v for u, v in zip(x, X)), sum(u * v for u, v in zip(x, Y))
        yX, yY = sum(u * v for u, v in zip(y, X)), sum(u * v for u, v in zip(y, Y))
        fp, fc = 0.5 * (xX * xX - xY * xY - yX * yX + yY * yY), xX * xY - yX * yY
        out.append((fp * 0.5 * (1.0 + ci * ci), -fc * ci, -(r[0] * cd * cp + r[1] * cd * sp + r[2] * sd) / CLIGHT))
    return out


def _strain(theta, f, n_det, gmst):
    """Detector strains [n_det][K] of one parameter set (11 floats)."""
    t = torch.tensor(theta, dtype=torch.float64, device="cuda")
    turns = (_coeffs(t[MC], t[Q], t[CHI1], t[CHI2], t[TC], t[PHIC])[:, None] * _basis(f)).sum(0)
    amp = _amplitude(t[MC], t[DL]) * f ** (-7.0 / 6.0) * (f < _isco(t[MC], t[Q]))
    rows = []
    for pr, pim, dt in _responses(t[RA], t[DEC], t[PSI], t[IOTA], gmst, n_det):
        ang = -2.0 * math.pi * torch.frac(turns + f * dt)
        rows.append(amp * torch.complex(pr, pim) * torch.polar(torch.ones_like(ang), ang))
    return torch.stack(rows)


def _event(family, df, n_det, seed, c128):
    """One synthetic event of a family and its Gaussian proposal in the Fisher metric."""
    fam = FAMILY[family]
    r = np.random.Generator(np.random.PCG64([seed, 11]))
    k = _n_bins(family, df)
    f = F_LO + df * torch.arange(k, dtype=torch.float64, device="cuda")
    psd = _psd(f)
    m = np.sort(r.uniform(*fam["m"], size=2))[::-1]
    th = np.zeros(11)
    th[MC] = (m[0] * m[1]) ** 0.6 / (m[0] + m[1]) ** 0.2
    th[Q] = m[0] / m[1]
    th[CHI1:CHI2 + 1] = r.uniform(-fam["chi"], fam["chi"], size=2)
    th[RA], th[DEC] = r.uniform(0, 2 * math.pi), math.asin(r.uniform(-1, 1))
    th[PSI], th[IOTA] = r.uniform(0, math.pi), math.acos(r.uniform(-1, 1))
    th[PHIC] = r.uniform(0, 2 * math.pi)
    gmst = r.uniform(0, 2 * math.pi)
    th[DL] = 1.0
    h = _strain(th, f, n_det, gmst)
    rho1 = math.sqrt(float((4 * df * h.abs() ** 2 / psd).sum()))
    th[DL] = rho1 / r.uniform(*fam["snr"])
    noise = torch.from_numpy(r.standard_normal((n_det, k, 2))).to("cuda")
    data = h / th[DL] + torch.view_as_complex(noise) * torch.sqrt(psd / (4 * df))
    data = data.to(torch.complex128 if c128 else torch.complex64)
    prop = _proposal(fam, th, f, df, n_det, gmst, psd)
    return dict(family=family, theta0=th, gmst=gmst, f=f, df=df, psd=psd, data=data, n_det=n_det, prop=prop)


def _proposal(fam, th, f, df, n_det, gmst, psd):
    """N(theta0, scale^2 Gamma^-1): marginalised slots projected out, weak widths where the
    data say little, and the prior box."""
    ids = fam["ids"]
    marg = [PHIC] * bool(fam["marg"] & mbis.MARG_PHASE) + [DL] * bool(fam["marg"] & mbis.MARG_DISTANCE)
    step = {MC: 1e-6 * th[MC], DL: 1e-5 * th[DL], CHI1: 1e-5, CHI2: 1e-5, TC: 1e-7}
    dh = []
    for p in ids + marg:
        s = step.get(p, 1e-6)
        up, dn = th.copy(), th.copy()
        up[p] += s
        dn[p] -= s
        dh.append((_strain(up, f, n_det, gmst) - _strain(dn, f, n_det, gmst)) / (2 * s))
    dh = torch.view_as_real(torch.stack(dh) * torch.sqrt(4 * df / psd)).reshape(len(dh), -1)
    g = (dh @ dh.T).cpu().numpy()
    P = len(ids)
    if marg:
        g = g[:P, :P] - g[:P, P:] @ np.linalg.solve(g[P:, P:], g[P:, :P])
    chi = fam["chi"]
    width = {Q: 2.0, CHI1: 2 * chi, CHI2: 2 * chi, RA: 2 * math.pi, DEC: math.pi, PSI: math.pi, IOTA: math.pi,
             PHIC: 2 * math.pi, DL: DMAX - DMIN}
    for i, p in enumerate(ids):
        if p in width:
            g[i, i] += 12.0 / width[p] ** 2
    cov = np.linalg.inv(g)
    chol = np.linalg.cholesky(0.5 * (cov + cov.T))
    lo, hi = np.zeros(P), np.zeros(P)
    fixed = {CHI1: (-chi, chi), CHI2: (-chi, chi), RA: (0, 2 * math.pi), DEC: (-math.pi / 2, math.pi / 2),
             PSI: (0, math.pi), IOTA: (0, math.pi), DL: (DMIN, DMAX), PHIC: (0, 2 * math.pi)}
    for i, p in enumerate(ids):
        if p in fixed:
            lo[i], hi[i] = fixed[p]
        else:
            d = 10.0 * fam["scale"] * math.sqrt(cov[i, i])
            lo[i], hi[i] = th[p] - d, th[p] + d
    i = ids.index(Q)
    lo[i] = max(lo[i], 1.0)
    i = ids.index(MC)
    lo[i] = max(lo[i], 0.1 * th[MC])
    return dict(ids=np.array(ids, np.int32), mean=th[ids].copy(), chol=chol, scale=fam["scale"], lo=lo, hi=hi,
                flags=fam["flags"])


def _samples(ev, n, seed):
    """n points of the event's proposal, [P][n], wrapped where a slot is periodic."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    p = ev["prop"]
    z = torch.randn((len(p["ids"]), n), dtype=torch.float64, device="cuda", generator=g)
    th = _dev(p["mean"])[:, None] + p["scale"] * (_dev(p["chol"]) @ z)
    for i, s in enumerate(p["ids"]):
        if s in (RA, PHIC, PSI):
            th[i] = torch.remainder(th[i], math.pi if s == PSI else 2 * math.pi)
    return th.contiguous()


# ---------------------------------------------------------------------------- the states

def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def _empty(*shape):
    return torch.empty(shape, dtype=torch.float64, device="cuda")


class _Handles:
    """Library objects of a state, destroyed with it."""

    def __init__(self):
        self.ctx, self.batch, self.tiling = [], None, None

    def __del__(self):
        if self.batch is not None:
            mbis.mbis_batch_destroy(self.batch)
        for c in self.ctx:
            mbis.mbis_destroy(c)
        if self.tiling is not None:
            mbis.mbis_tiling_destroy(self.tiling)


class _Borrowed:
    """A device buffer of the library as an array that torch can read; keeps its owner alive."""

    def __init__(self, ptr, shape, owner):
        self.owner = owner
        self.__cuda_array_interface__ = dict(shape=shape, typestr="<f8", data=(ptr, False), version=3)


def _context(ev, precision, handles):
    fam = FAMILY[ev["family"]]
    sites = SITES[:ev["n_det"]]
    dets = mbis.make_detectors([s[0] for s in sites], [s[1] for s in sites], [s[2] for s in sites])
    psd = np.broadcast_to(ev["psd"].cpu().numpy(), (ev["n_det"], len(ev["f"])))
    ctx = mbis.mbis_create(ev["data"].cpu().numpy(), psd, dets, F_LO, ev["df"], ev["theta0"], gmst=ev["gmst"],
                           precision=mbis.FP64 if precision == "fp64" else mbis.MIXED, marg=fam["marg"],
                           n_tshift=N_SHIFT, dt_shift=DT_SHIFT, dmin=DMIN, dmax=DMAX)
    handles.ctx.append(ctx)
    p = ev["prop"]
    mbis.mbis_set_metric(ctx, p["ids"], p["mean"], p["chol"], p["scale"], p["lo"], p["hi"], p["flags"])
    return ctx


def _batch_plan(case):
    """Family, bin spacing, detectors and samples of each event of a batch."""
    dfs = [1 / 4, 1 / 128, 1 / 16, 1 / 32, 1 / 64, 1 / 8]
    return [("bns" if i % 2 else "heavy", dfs[i % 6], 2 + (i // 2) % 2,
             (1 << case["log2_n"] + (3 * i) % 4) - (37 * i if i % 3 == 2 else 0)) for i in range(case["events"])]


def _stage_inputs(case, seed):
    """Samples of a refitted proposal: log L about a narrower Gaussian than the proposal, some
    points outside the prior, and the point whose levels are asked."""
    n, P = case["n"], case["p"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn((P, n), dtype=torch.float64, device="cuda", generator=g)
    r = np.random.Generator(np.random.PCG64([seed, 12]))
    mean, chol = r.uniform(0.5, 1.2, P), np.tril(r.normal(0, 0.05, (P, P)), -1) + np.diag(r.uniform(0.05, 0.2, P))
    theta = (_dev(mean)[:, None] + _dev(chol) @ z).contiguous()
    tilt = _dev(r.uniform(0.95, 1.6, P))
    loglike = 180.0 - 0.5 * ((z - 0.2) ** 2 * tilt[:, None]).sum(0)
    log_q = -0.5 * (z * z).sum(0)
    log_prior = torch.where(z[0].abs() < 2.5, 0.4 * z[-1], torch.full_like(z[0], -math.inf))
    return theta, loglike, log_prior, log_q, mean, chol, mean + 0.05 * r.normal(size=P)


def _candidates(n, seed):
    r = np.random.Generator(np.random.PCG64([seed, 13]))
    return np.stack([r.uniform(SPACE["x_lo"], SPACE["x_hi"], n), r.uniform(SPACE["q_lo"], SPACE["q_hi"], n)])


BANK = dict(n=1 << 15, min_match=0.99, stop_after=1000, most=1024)


def _tile_points(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    u = torch.rand((2, case["n"]), dtype=torch.float64, device="cuda", generator=g)
    lo = _dev([SPACE["x_lo"], SPACE["q_lo"]])[:, None]
    hi = _dev([SPACE["x_hi"], SPACE["q_hi"]])[:, None]
    return (lo + (hi - lo) * u).contiguous()


def prepare(case, seed):
    kind, hold = case["kind"], _Handles()
    st = dict(case=case, hold=hold, seed=seed)
    if kind in ("loglike", "pass"):
        ev = _event(case["family"], case["df"], case["det"], seed, case["c128"])
        st["ctx"], n, P = _context(ev, case["precision"], hold), case["n"], len(ev["prop"]["ids"])
        st["loglike"] = _empty(n)
        if kind == "loglike":
            st["theta"] = _samples(ev, n, seed)
        else:
            st.update(theta=_empty(P, n), log_q=_empty(n), log_prior=_empty(n), weights=_empty(n))
    elif kind == "draw":
        ev = _event(case["family"], 0.25, 2, seed, False)
        n, P = case["n"], len(ev["prop"]["ids"])
        st.update(ctx=_context(ev, "fp64", hold), theta=_empty(P, n), log_q=_empty(n), log_prior=_empty(n))
    elif kind == "batch":
        plan = _batch_plan(case)
        evs = [_event(f, df, det, 1000 * seed + i, False) for i, (f, df, det, _) in enumerate(plan)]
        ctxs = [_context(ev, "mixed", hold) for ev in evs]
        ns = [p[3] for p in plan]
        hold.batch = mbis.mbis_batch_create(ctxs, ns, [seed + 100 + i for i in range(len(ns))])
        st["loglike"] = [torch.as_tensor(_Borrowed(mbis.mbis_batch_buffers(hold.batch, i)[1], (n,), hold), device="cuda")
                         for i, n in enumerate(ns)]
    elif kind == "ess":
        ev = _event(case["family"], case["df"], case["det"], seed, False)
        ctx = _context(ev, "mixed", hold)
        edges = mbis.mbis_rb_edges(ctx, ev["theta0"], 5.0, 0.3)
        mbis.mbis_rb_setup(ctx, ev["theta0"], edges)
        mbis.mbis_rb_use(ctx)
        n, P = case["batch"], len(ev["prop"]["ids"])
        st.update(ctx=ctx, prop=ev["prop"], theta=_empty(P, n), log_q=_empty(n), log_prior=_empty(n),
                  loglike=_empty(n), weights=_empty(n))
    elif kind == "stage":
        theta, ll, lp, lq, mean, chol, ref = _stage_inputs(case, seed)
        # a context over the same slots carries the proposal the moments are taken about
        family = {2: "heavy", 4: "heavy", 5: "bns", 11: "bbh"}[case["p"]]
        ev = _event(family, 0.25, 2, seed, False)
        ctx = _context(ev, "fp64", hold)
        ids = ev["prop"]["ids"][:case["p"]]
        lo, hi = np.full(len(ids), 0.01), np.full(len(ids), 1.5)
        mbis.mbis_set_metric(ctx, ids, mean, chol, 1.0, lo, hi, 0)
        st.update(ctx=ctx, theta=theta, loglike=ll, log_prior=lp, log_q=lq, ref=ref, weights=_empty(case["n"]),
                  levels=_empty(case["p"]))
    elif kind == "tiles":
        k = int((TILE_F_HI - F_LO) / TILE_DF) + 1
        f = F_LO + TILE_DF * torch.arange(k, dtype=torch.float64, device="cuda")
        t = mbis.mbis_tiling_create(F_LO, TILE_DF, k, _psd(f).cpu().numpy(), **SPACE)
        hold.tiling = t
        mbis.mbis_tiling_bank(t, _candidates(BANK["n"], seed), BANK["min_match"], BANK["stop_after"], BANK["most"])
        st.update(points=_tile_points(case, seed), tile=torch.empty(case["n"], dtype=torch.int32, device="cuda"),
                  match=torch.empty(case["n"], dtype=torch.float32, device="cuda"))
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "loglike":
        mbis.mbis_loglike(st["ctx"], case["n"], st["theta"], st["loglike"])
        return st["loglike"]
    if kind == "draw":
        mbis.mbis_draw(st["ctx"], st["seed"], 0, case["n"], st["theta"], st["log_q"], st["log_prior"])
        return st["theta"], st["log_q"], st["log_prior"]
    if kind == "pass":
        c, n = st["ctx"], case["n"]
        mbis.mbis_draw(c, st["seed"], 0, n, st["theta"], st["log_q"], st["log_prior"])
        mbis.mbis_loglike(c, n, st["theta"], st["loglike"])
        s = mbis.mbis_reduce(c, n, st["loglike"], st["log_prior"], st["log_q"], st["weights"])
        return dict(theta=st["theta"], log_q=st["log_q"], log_prior=st["log_prior"], loglike=st["loglike"],
                    weights=st["weights"], ess=s["ess"], log_z=s["log_z"])
    if kind == "batch":
        s = mbis.mbis_batch_step(st["hold"].batch, 1, case["events"])
        return dict(loglike=st["loglike"], ess=np.array([x["ess"] for x in s]),
                    log_z=np.array([x["log_z"] for x in s]))
    if kind == "ess":
        p = st["prop"]
        mbis.mbis_set_proposal(st["ctx"], p["mean"], p["chol"], p["scale"])
        s, drawn, used = mbis.mbis_run_to_ess(st["ctx"], st["theta"], st["log_q"], st["log_prior"], st["loglike"],
                                              st["weights"], 1e4, case["batch"], 16 * case["batch"], st["seed"],
                                              refine=4, refine_scale=1.2)
        mean, chol, _ = mbis.mbis_get_proposal(st["ctx"], len(p["ids"]))
        return dict(ess=s["ess"], log_z=s["log_z"], drawn=drawn, used=used, mean=mean, chol=chol)
    if kind == "stage":
        n = case["n"]
        s = mbis.mbis_reduce(st["ctx"], n, st["loglike"], st["log_prior"], st["log_q"], st["weights"])
        mean, cov = mbis.mbis_weighted_moments(st["ctx"], n, st["theta"], st["weights"])
        mbis.mbis_credible_levels(n, st["theta"], st["weights"], st["ref"], st["levels"])
        return dict(weights=st["weights"], ess=s["ess"], log_z=s["log_z"], mean=mean, cov=cov, levels=st["levels"])
    mbis.mbis_tiling_assign(st["hold"].tiling, case["n"], st["points"], st["tile"], st["match"])
    return st["tile"], st["match"]


# ---------------------------------------------------------------------------- what a pass needs

def _loglike_work(family, df, det, n):
    k, P = _n_bins(family, df), len(FAMILY[family]["ids"])
    rows = det if family == "bbh" else 1
    # the bins below the ISCO of the family's typical total mass: the others are zero
    k = min(k, int(((4397.0 / {"heavy": 60.0, "bns": 3.1}.get(family, 70.0)) - F_LO) / df))
    # per sample, bin and table row: a nine-term phase, a sine, a cosine and a complex
    # multiply-add; per sample and bin the 128 time shifts where they are marginalised
    flops = n * k * (rows * (18 + 2 + 8) + (4 * N_SHIFT if family == "bbh" else 0))
    return 8.0 * n * (P + 1) + 8.0 * k * rows, float(flops)


def work(case):
    kind = case["kind"]
    if kind == "loglike":
        b, f = _loglike_work(case["family"], case["df"], case["det"], case["n"])
    elif kind == "pass":
        b, f = _loglike_work(case["family"], case["df"], case["det"], case["n"])
        b += 8.0 * case["n"] * 8
    elif kind == "draw":
        P = len(FAMILY[case["family"]]["ids"])
        b, f = 8.0 * case["n"] * (P + 2), case["n"] * (60.0 * P + P * P)
    elif kind == "batch":
        parts = [_loglike_work(f, df, det, n) for f, df, det, n in _batch_plan(case)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "ess":
        # at least five batches (four of them refits); about 1300 coarse bins per sample
        b, f = 5 * 8.0 * case["batch"] * 9, 5 * 28.0 * 1300 * case["batch"]
    elif kind == "stage":
        b, f = 8.0 * case["n"] * (3 + 1 + 2 * (case["p"] + 1)), case["n"] * (60.0 + 2.0 * case["p"] ** 2)
    else:
        # eight operations per point, live bin (about 200 of 433) and template (about 340)
        b, f = 24.0 * case["n"], 8.0 * 200 * 340 * case["n"]
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------------------- 64-bit answers

def _log_i0(x):
    return torch.log(torch.special.i0e(x)) + x


def _exact_distance(z1, h1):
    """ln int p(d) I0(Z1/d) e^(-H1/(2 d^2)) dd by 64 panels of 16 Gauss-Legendre points in ln d."""
    x, w = np.polynomial.legendre.leggauss(16)
    a, b, panels = -math.log(DMAX), -math.log(DMIN), 64
    half = 0.5 * (b - a) / panels
    s = _dev((a + half * (2 * np.arange(panels)[:, None] + 1 + x)).reshape(-1))
    lw = _dev(np.log(np.tile(half * w, panels)))
    c0 = math.log(3.0 / (DMAX ** 3 - DMIN ** 3))
    out = []
    for z, h in zip(z1.split(8192), h1.split(8192)):
        u = torch.exp(s)
        out.append(torch.logsumexp(c0 - 3 * s + lw + _log_i0(z[:, None] * u) - 0.5 * h[:, None] * u * u, 1))
    return torch.cat(out)


def _exact_loglike(ev, theta):
    """log L of samples [P][n] by the plain sum over bins and detectors, in 64 bits."""
    fam, f, df = FAMILY[ev["family"]], ev["f"], ev["df"]
    n, full = theta.shape[1], [None] * 11
    for s in range(11):
        full[s] = torch.full((theta.shape[1],), float(ev["theta0"][s]), dtype=torch.float64, device="cuda")
    for i, s in enumerate(ev["prop"]["ids"]):
        full[s] = theta[i]
    if fam["marg"] & mbis.MARG_PHASE:
        full[PHIC] = torch.zeros(n, dtype=torch.float64, device="cuda")
    if fam["marg"] & mbis.MARG_DISTANCE:
        full[DL] = torch.ones(n, dtype=torch.float64, device="cuda")
    f_max = float(_isco(full[MC], full[Q]).nan_to_num(0.0).max())
    k = max(1, int((f < f_max).sum()))
    f = f[:k]
    basis = _basis(f)
    data = ev["data"][:, :k].to(torch.complex128)
    amp76 = f ** (-7.0 / 6.0)
    wt = 4 * df * data.conj() * amp76 / ev["psd"][:k]
    norm = 4 * df * amp76 ** 2 / ev["psd"][:k]
    tau = (torch.arange(N_SHIFT, dtype=torch.float64, device="cuda") - N_SHIFT // 2) * DT_SHIFT
    if fam["marg"] == mbis.MARG_TIME:
        turn = torch.frac(f[:, None] * tau)
        tw = torch.cat([torch.cos(2 * math.pi * turn), torch.sin(2 * math.pi * turn)])
    out = []
    step = max(1, (1 << 25) // k)
    for c in range(0, n, step):
        p = [v[c:c + step] for v in full]
        turns = _coeffs(p[MC], p[Q], p[CHI1], p[CHI2], p[TC], p[PHIC]).T @ basis
        live = f < _isco(p[MC], p[Q])[:, None]
        A = _amplitude(p[MC], p[DL])
        hsum = (live * norm).sum(1)
        zr = zi = 0.0
        h = 0.0
        for d, (pr, pim, dt) in enumerate(_responses(p[RA], p[DEC], p[PSI], p[IOTA], ev["gmst"], ev["n_det"])):
            ang = 2 * math.pi * torch.frac(turns + dt[:, None] * f)
            co, si = torch.cos(ang) * live, torch.sin(ang) * live
            wr, wi = wt[d].real, wt[d].imag
            if fam["marg"] == mbis.MARG_TIME:
                # a_k = w e^(-i ang) P
                ar, ai = co * wr + si * wi, co * wi - si * wr
                zr = zr + pr[:, None] * ar - pim[:, None] * ai
                zi = zi + pr[:, None] * ai + pim[:, None] * ar
            else:
                ar, ai = co @ wr + si @ wi, co @ wi - si @ wr
                zr, zi = zr + pr * ar - pim * ai, zi + pr * ai + pim * ar
            h = h + (pr * pr + pim * pim) * hsum
        h = A * A * h
        if fam["marg"] == mbis.MARG_TIME:
            zj = A[:, None] * (torch.cat([zr, zi], 1) @ tw)
            ll = torch.logsumexp(zj, 1) - math.log(N_SHIFT) - 0.5 * h
        elif fam["marg"] & mbis.MARG_DISTANCE:
            ll = _exact_distance(A * torch.hypot(zr, zi), h)
        else:
            ll = _log_i0(A * torch.hypot(zr, zi)) - 0.5 * h
        out.append(ll)
    ll = torch.cat(out)
    bad = ~(full[MC] > 0) | ~(full[Q] > 0) | ~(full[CHI1].abs() < 1) | ~(full[CHI2].abs() < 1) | ~(full[DL] > 0)
    return torch.where(bad, torch.full_like(ll, -math.inf), ll)


def _philox(ctr, tag, block, seed):
    """Philox4x32-10 words (int64 tensors) of counters (lo, hi, tag, block) and the key's halves."""
    m32 = 0xFFFFFFFF
    c = [ctr & m32, ctr >> 32, torch.full_like(ctr, tag), torch.full_like(ctr, block)]
    k0, k1 = seed & m32, (seed >> 32) & m32

    def mul(a, x):  # 32 x 32 -> (high, low) in pieces that fit 63 bits
        lo, hi = a & 0xFFFF, a >> 16
        low = x * lo
        t = x * hi + (low >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (low & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c


def _exact_draw(prop, seed, ctr0, n):
    ids, P = prop["ids"], len(prop["ids"])
    ctr = ctr0 + torch.arange(n, dtype=torch.int64, device="cuda")
    z = []
    for blk in range((P + 3) // 4):
        w = [(v.double() + 0.5) * INV_2_32 for v in _philox(ctr, 2, blk, seed)]
        for a, b in ((w[0], w[1]), (w[2], w[3])):
            r = torch.sqrt(-2.0 * torch.log(a))
            z += [r * torch.cos(2 * math.pi * b), r * torch.sin(2 * math.pi * b)]
    z = torch.stack(z[:P])
    chol = _dev(prop["chol"])
    theta = _dev(prop["mean"])[:, None] + prop["scale"] * (chol @ z)
    log_q = -0.5 * (z * z).sum(0) - float(np.log(np.diag(prop["chol"])).sum()) - 0.5 * P * math.log(2 * math.pi) \
        - P * math.log(prop["scale"])
    lp = torch.zeros(n, dtype=torch.float64, device="cuda")
    inside = torch.ones(n, dtype=torch.bool, device="cuda")
    m1m2 = bool(prop["flags"] & mbis.PRIOR_M1M2)
    box = {}
    for i, s in enumerate(ids):
        lo, hi = float(prop["lo"][i]), float(prop["hi"][i])
        box[int(s)] = (lo, hi)
        if s in (RA, PHIC, PSI):
            period = math.pi if s == PSI else 2 * math.pi
            theta[i] = torch.remainder(theta[i], period)
            lp -= math.log(period)
            continue
        x = theta[i]
        inside &= (x >= lo) & (x <= hi)
        if s == DEC:
            lp += torch.log(torch.cos(x)) - math.log(math.sin(hi) - math.sin(lo))
        elif s == IOTA:
            lp += torch.log(torch.sin(x)) - math.log(math.cos(lo) - math.cos(hi))
        elif s == DL:
            lp += 2 * torch.log(x) + math.log(3.0) - math.log(hi ** 3 - lo ** 3)
        elif not (m1m2 and s in (MC, Q)):
            lp -= math.log(hi - lo)
    if m1m2:
        mc, q = theta[list(ids).index(MC)], theta[list(ids).index(Q)]
        x, w = np.polynomial.legendre.leggauss(200)
        (ml, mh), (ql, qh) = box[MC], box[Q]
        qq = 0.5 * (qh + ql) + 0.5 * (qh - ql) * x
        norm = 0.5 * (mh ** 2 - ml ** 2) * 0.5 * (qh - ql) * float((w * (1 + qq) ** 0.4 * qq ** -1.2).sum())
        lp += torch.log(mc) + 0.4 * torch.log(1 + q) - 1.2 * torch.log(q) - math.log(norm)
    return theta, log_q, torch.where(inside, lp, torch.full_like(lp, -math.inf))


def _exact_weights(ll, lp, lq):
    lw = ll + lp - lq
    m = lw.max()
    e = torch.where(torch.isfinite(lw), torch.exp(lw - m), torch.zeros_like(lw))
    s1, s2 = e.sum(), (e * e).sum()
    return e / s1, float(s1 * s1 / s2), float(m + torch.log(s1)) - math.log(len(lw))


def _exact_tiles(case, seed):
    """The best match of every point with the templates of the bank, the bank placed in order."""
    k = int((TILE_F_HI - F_LO) / TILE_DF) + 1
    f = F_LO + TILE_DF * torch.arange(k, dtype=torch.float64, device="cuda")
    basis, w = _basis(f), f ** (-7.0 / 6.0) / torch.sqrt(_psd(f))

    def waveforms(x, q):
        mc = SPACE["mc_base"] + torch.remainder(x, SPACE["mc_period"])
        q = torch.where(q >= 1, q, 1 / q)
        zero = torch.zeros_like(mc)
        turns = torch.frac(_coeffs(mc, q, zero, zero, zero, zero).T @ basis)
        a = w * (f < _isco(mc, q)[:, None])
        return torch.polar(a / torch.linalg.vector_norm(a, dim=1, keepdim=True), -2 * math.pi * turns)

    cand = _dev(_candidates(BANK["n"], seed))
    bank, rejected, T = torch.empty((0, k), dtype=torch.complex128, device="cuda"), 0, 0
    for c in range(0, BANK["n"], 256):
        u = waveforms(cand[0, c:c + 256], cand[1, c:c + 256])
        best = (u.conj() @ bank.T).abs().max(1).values.cpu().numpy() if T else np.zeros(len(u))
        inner = (u.conj() @ u.T).abs().cpu().numpy()
        keep = []
        for i in range(len(u)):
            if max(best[i], max((inner[i, j] for j in keep), default=0.0)) < BANK["min_match"]:
                keep.append(i)
                T, rejected = T + 1, 0
            else:
                rejected += 1
            if rejected >= BANK["stop_after"] or T >= BANK["most"]:
                break
        bank = torch.cat([bank, u[keep]])
        if rejected >= BANK["stop_after"] or T >= BANK["most"]:
            break
    pts, out = _tile_points(case, seed), []
    for x, q in zip(pts[0].split(16384), pts[1].split(16384)):
        out.append((waveforms(x, q).conj() @ bank.T).abs().max(1).values)
    return torch.cat(out)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("loglike", "pass"):
        if case["n"] * _n_bins(case["family"], case["df"]) > 5e10:
            return None  # minutes in 64 bits
        ev = _event(case["family"], case["df"], case["det"], seed, case["c128"])
        if kind == "loglike":
            return _exact_loglike(ev, _samples(ev, case["n"], seed))
        theta, lq, lp = _exact_draw(ev["prop"], seed, 0, case["n"])
        ll = _exact_loglike(ev, theta)
        w, ess, log_z = _exact_weights(ll, lp, lq)
        return dict(theta=theta, log_q=lq, log_prior=lp, loglike=ll, weights=w, ess=ess, log_z=log_z)
    if kind == "draw":
        ev = _event(case["family"], 0.25, 2, seed, False)
        return _exact_draw(ev["prop"], seed, 0, case["n"])
    if kind == "batch":
        ll, ess, log_z = [], [], []
        for i, (f, df, det, n) in enumerate(_batch_plan(case)):
            ev = _event(f, df, det, 1000 * seed + i, False)
            theta, lq, lp = _exact_draw(ev["prop"], seed + 100 + i, n, n)
            ll.append(_exact_loglike(ev, theta))
            _, e, z = _exact_weights(ll[-1], lp, lq)
            ess.append(e)
            log_z.append(z)
        return dict(loglike=ll, ess=np.array(ess), log_z=np.array(log_z))
    if kind == "ess":
        return None  # the result of a loop whose proposals depend on every earlier batch
    if kind == "stage":
        theta, ll, lp, lq, mean, _, ref = _stage_inputs(case, seed)
        w, ess, log_z = _exact_weights(ll, lp, lq)
        family = {2: "heavy", 4: "heavy", 5: "bns", 11: "bbh"}[case["p"]]
        period = {RA: 2 * math.pi, PHIC: 2 * math.pi, PSI: math.pi}
        per = [period.get(s, 0.0) for s in FAMILY[family]["ids"][:case["p"]]]
        d = theta - _dev(mean)[:, None]
        for i, t in enumerate(per):
            if t:
                d[i] -= t * torch.floor(d[i] / t + 0.5)
        off = (w * d).sum(1)
        cov = (w * d) @ d.T - off[:, None] * off
        m = (_dev(mean) + off).cpu().numpy()
        m = np.array([x - t * math.floor(x / t) if t else x for x, t in zip(m, per)])
        levels = ((theta < _dev(ref)[:, None]) * w).sum(1) + 0.5 * ((theta == _dev(ref)[:, None]) * w).sum(1)
        return dict(weights=w, ess=ess, log_z=log_z, mean=m, cov=cov, levels=levels)
    return None, _exact_tiles(case, seed)
