"""The work that a user of paper_2607_24141_gb300 has it do, as cases that can be timed.

Every case goes through the package's public calls: a Synthesizer is made once (``prepare``)
and ``run`` makes one pass on it -- a forward synthesis, a forward with its reverse pass, or
one evaluation of a calibration.  Sizes are those of the package's own configurations
(``inputs.config0`` .. ``config4_joint_grouped``), of its smoke test and of its scaling sweep,
or scaled variants of them.

``exact`` computes the same outputs in FP64 with torch alone: the windowed Voigt sum line by
line, the closed-form transfer, the instrument's weights and (by automatic differentiation
from the opacity on, by the definition below it) the gradients.
"""
import math

import numpy as np
import torch

import paper_2607_24141_gb300 as pz
from paper_2607_24141_gb300 import inputs as I

H_BAND = (1500.0, 1700.0)     # the H-band window of the package's configurations, nm
N_ELEM = 20                   # elements of the H-band species
OPTICAL = ("solar", "solar_fp64", "optical")
FORWARD = OPTICAL + ("forward",)


def listed():
    return [
        # one small window around a few lines, fitted through torch autograd: the smallest
        # call, where launches and host work count (the smoke test's size)
        dict(name="window_autograd", kind="autograd", lam_lo=1600.0, span=6.398, lines=60, bands=0, W=300),
        # the 4,000-point solar optical spectrum (configuration 0), forward only
        dict(name="tiny_forward", kind="solar", points=4000, lines=2000, W=1000),
        # the same kind of spectrum in the plain FP64 form, the check of a mixed result
        dict(name="solar_fp64", kind="solar_fp64", points=1019, lines=600, W=300),
        # a 12 nm piece of an H-band fit at full line density, with odd sizes: fwd, chi^2, bwd
        dict(name="piece_step", kind="step", lam_lo=1590.0, span=11.77, lines=11973, bands=0, W=1500, eta=0.0),
        # the APOGEE-like spectrum (configuration 1): synthesis alone ...
        dict(name="hband_forward", kind="forward", lam_lo=1500.0, span=200.0, lines=133500, bands=133, W=1500, eta=0.0),
        # ... and with objective and gradients
        dict(name="hband_step", kind="step", lam_lo=1500.0, span=200.0, lines=133500, bands=133, W=1500, eta=0.0),
        # the same step with the continuum-referenced centre test, as production synthesis runs
        dict(name="hband_centre_step", kind="step", lam_lo=1500.0, span=200.0, lines=133500, bands=133, W=1500,
             eta=1e-3),
        # an evaluation of the two-star calibration with per-line corrections (one graph launch)
        dict(name="joint_calibration", kind="joint", lines=100000),
        # an evaluation of the grouped four-parameter calibration (42,886 records)
        dict(name="grouped_calibration", kind="group", complexes=25281, records=42886),
        # a broad optical synthesis at full resolution, the densest part of configuration 2
        dict(name="broad_forward", kind="optical", lam_lo=300.0, span=100.0, lines=1071429, W=2000, R=3e5, eta=0.0),
        # H-band piece with continuum scattering, fwd and bwd
        dict(name="scatter_step", kind="scatter_step", lam_lo=1600.0, span=8.0, lines=5337, bands=0, W=1500, eta=0.0),
        # a batch of stars on one list, one calibration evaluation (the benchmark's recipe)
        dict(name="batch_calibration", kind="batch", stars=8, scale=0.6),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["autograd", "solar", "optical", "optical", "solar_fp64", "forward", "step", "step", "joint", "group",
                       "scatter_step", "batch"])
    if kind == "autograd":
        span = _log(rng, 1.5, 25.0)
        return dict(kind=kind, lam_lo=rng.uniform(1510.0, 1660.0), span=span, lines=int(_log(rng, 20, 700 * span)),
                    bands=0, W=int(_log(rng, 100, 2000)))
    if kind == "optical":
        # sampling from a tenth of full resolution up; windows keep their width in wavelength
        R = rng.choice([1e4, 3e4, 1e5, 3e5, 3e5, 3e5]) * rng.uniform(0.9, 1.1)
        lam = rng.uniform(300.0, 800.0)
        span = _log(rng, 2.0, 100.0)
        W = max(20, int(2000 * R / 3e5 * rng.uniform(0.5, 1.05)))
        lines = int(span * _log(rng, 100, 4000))
        return dict(kind=kind, lam_lo=lam, span=span, lines=lines, W=W, R=R, eta=rng.choice([0.0, 0.0, 1e-3]))
    if kind == "solar":
        n = int(_log(rng, 500, 12000))
        return dict(kind=kind, points=n, lines=int(n * _log(rng, 0.05, 2.0)) + 1, W=int(_log(rng, 60, 2000)))
    if kind == "solar_fp64":
        return dict(kind=kind, points=int(_log(rng, 200, 1200)), lines=int(_log(rng, 100, 900)),
                    W=int(_log(rng, 50, 400)))
    if kind in ("forward", "step"):
        span = _log(rng, 3.0, 180.0)
        lo = rng.uniform(H_BAND[0], H_BAND[1] - span)
        return dict(kind=kind, lam_lo=lo, span=span, lines=int(span * _log(rng, 60, 1300)),
                    bands=int(rng.uniform(0, 0.7) * span) if span > 20 else 0, W=int(_log(rng, 300, 2000)),
                    eta=rng.choice([0.0, 0.0, 1e-3]))
    if kind == "joint":
        return dict(kind=kind, lines=int(_log(rng, 2e4, 1.5e5)))
    if kind == "group":
        n = int(_log(rng, 6e3, 3e4))
        return dict(kind=kind, complexes=n, records=int(n * rng.uniform(1.2, 2.2)))
    if kind == "scatter_step":
        span = _log(rng, 2.0, 12.0)
        return dict(kind=kind, lam_lo=rng.uniform(1510.0, 1680.0), span=span, lines=int(span * _log(rng, 60, 700)),
                    bands=0, W=int(_log(rng, 300, 2000)), eta=0.0)
    return dict(kind=kind, stars=rng.choice([2, 3, 4, 5, 6]), scale=rng.uniform(0.1, 0.6))


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------

def _problem(case, seed):
    """The Problem or Batch of a case (host arrays)."""
    k = case["kind"]
    if k in ("solar", "solar_fp64"):
        return I.config0(seed=seed, n_lambda=case["points"], n_lines=case["lines"], W=case["W"])
    if k == "optical":
        lo = case["lam_lo"]
        return I.config2(seed=seed, lam_lo=lo, lam_hi=lo + case["span"], n_lines=case["lines"], W=case["W"], R=case["R"])
    if k in ("autograd", "forward", "step", "scatter_step"):
        lo, hi = case["lam_lo"], case["lam_lo"] + case["span"]
        p = I.config1(seed=seed, lam_lo=lo, lam_hi=hi, n_bands=case["bands"], n_atomic=case["lines"], W=case["W"])
        if k == "scatter_step":
            p = I.with_scattering(p, r0=50.0)
        return p
    if k == "joint":
        return I.config4_joint(seed=seed, n_common=case["lines"])[0]
    if k == "group":
        return I.config4_joint_grouped(seed=seed, n_complexes=case["complexes"], n_records=case["records"])
    if k == "batch":
        return I.config4(seed=seed, n_stars=case["stars"], nk_scale=case["scale"])
    raise ValueError(k)


def _observed(rng, shape):
    """Synthetic observed spectra: blended absorption features and S/N 200 noise."""
    d = rng.exponential(0.06, shape)
    k = np.exp(-0.5 * (np.arange(-4, 5) / 1.6) ** 2)
    y = np.apply_along_axis(lambda v: np.convolve(v, k / k.sum(), "same"), -1, d)
    return (np.clip(1.0 - y, 0.02, 1.0) + rng.normal(0.0, 1.0 / 200.0, shape)).astype(np.float32)


def _corrections(rng, n, n_elem):
    """Corrections as a fit meets them midway: oscillator strengths, damping, abundances."""
    return (rng.normal(0.0, 0.1, n).astype(np.float32), rng.normal(0.0, 0.2, n).astype(np.float32),
            rng.normal(0.0, 0.05, n_elem).astype(np.float32))


def _host(case, seed):
    """(problem, observed spectra, corrections, extras) on the host, from the seed alone."""
    made = _problem(case, seed)
    prob, truth = made if isinstance(made, tuple) else (made, None)
    rng = np.random.default_rng(1_000_003 + seed)
    n_out = prob.instrument.pix_lambda_nm.size if prob.instrument is not None else prob.grid.n_lambda
    shape = (prob.n_stars, n_out) if hasattr(prob, "subsets") else (n_out,)
    y = _observed(rng, shape)
    w = np.full(shape, 200.0 ** 2, np.float32)
    w[rng.random(shape) < 0.03] = 0.0        # masked pixels
    corr = _corrections(rng, prob.lines.n_lines, N_ELEM)
    return prob, truth, y, w, corr


def prepare(case, seed):
    prob, truth, y, w, corr = _host(case, seed)
    k = case["kind"]
    dev = torch.device("cuda", 0)
    s = pz.Synthesizer(prob, pz.PZ_FP64 if k == "solar_fp64" else pz.PZ_MIXED)
    if case.get("eta"):
        pz.pz_set_centre_test(s.ctx, case["eta"])
    st = {"kind": k, "s": s}
    nl, n = s.n_lines, s.n_lambda
    f32 = dict(dtype=torch.float32, device=dev)
    if k in OPTICAL:
        st["kappa"] = torch.empty((s.n_depth, n), **f32)
    if k in FORWARD:
        st["F"] = torch.empty(n, dtype=torch.float64, device=dev)
        st["Fc"] = torch.empty(n, dtype=torch.float64, device=dev)
        st["f"] = torch.empty(s.n_out, **f32)
        return st
    st["y"], st["w"] = torch.from_numpy(y).to(dev), torch.from_numpy(w).to(dev)
    st["loss"] = torch.zeros(1, dtype=torch.float64, device=dev)
    if k == "group":
        # corrections linked within each complex of records
        q, G = truth["complex_of_line"], case["complexes"]
        s.forward()
        pz.pz_set_line_groups(s.ctx, q, G)
        st["x"] = torch.from_numpy(np.random.default_rng(seed).normal(0.0, 0.15, (4, G)).astype(np.float32)).to(dev)
        st["g"] = torch.empty((4, G), **f32)
        return st
    st["c"] = [torch.from_numpy(a).to(dev) for a in corr]
    if k == "autograd":
        for t in st["c"]:
            t.requires_grad_(True)
        return st
    st["g_gf"], st["g_g6"], st["g_ab"] = torch.empty(nl, **f32), torch.empty(nl, **f32), torch.empty(N_ELEM, **f32)
    if k in ("joint", "batch"):
        s.set_corrections(*st["c"])
        s.forward()                        # configures the instrument, as the calibration drivers ask
    else:
        st["f"] = torch.empty(s.n_out, **f32)
        st["dL"] = torch.empty(s.n_out, **f32)
    return st


def run(st):
    k, s = st["kind"], st["s"]
    if k in FORWARD:
        s.forward(st.get("kappa"), st["F"], st["Fc"], st["f"])
        out = {"F": st["F"], "Fc": st["Fc"], "f": st["f"]}
        if "kappa" in st:
            out["kappa"] = st["kappa"]
        return out
    if k == "autograd":
        f = pz.SynthesisFunction.apply(s, *st["c"])
        loss = (st["w"] * (f - st["y"]) ** 2).sum()
        g = torch.autograd.grad(loss, st["c"])
        return {"f": f, "loss": loss, "g_gf": g[0], "g_g6": g[1], "g_ab": g[2]}
    if k == "group":
        pz.pz_group_eval(s.ctx, st["y"], st["w"], st["x"], st["loss"], st["g"])
        return {"loss": st["loss"], "g": st["g"]}
    s.set_corrections(*st["c"])
    if k in ("joint", "batch"):
        s.calib_step(st["y"], st["w"], 0.0, 0.0, 0.0, st["loss"], st["g_gf"], st["g_g6"], st["g_ab"])
        return {"loss": st["loss"], "g_gf": st["g_gf"], "g_g6": st["g_g6"], "g_ab": st["g_ab"]}
    s.forward(f=st["f"])
    s.loss(st["y"], st["w"], st["loss"], st["dL"])
    s.backward(st["dL"], st["g_gf"], st["g_g6"], st["g_ab"])
    return {"f": st["f"], "loss": st["loss"], "dL": st["dL"], "g_gf": st["g_gf"], "g_g6": st["g_g6"], "g_ab": st["g_ab"]}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
# Bytes: per star and grid point the FP64 atmosphere tables of each layer (continuum, Planck,
# stimulated emission) once and the opacity once; per line its record and its outputs.
# Operations: the line profile has to be evaluated near each line's core (within 20 Doppler
# widths, about 1.9 km/s wide on average, at about 40 operations, 90 with its derivative), the
# strength and damping of every (line, layer) once (about 40), and two exponential integrals per
# (point, layer) and branch (56 each), a third with the reverse pass.  The far wings are smooth:
# a sum over them needs no term per (line, point).

def work(case):
    k = case["kind"]
    R = case.get("R", 3e5)
    lo, span = case.get("lam_lo", H_BAND[0]), case.get("span", H_BAND[1] - H_BAND[0])
    n = case.get("points", int(math.log((lo + span) / lo) * R) + 1)
    stars, nd = 1, 72
    lines = case.get("lines", 0) + 500 * case.get("bands", 0)
    if k == "joint":
        stars = 2
    elif k == "group":
        stars, lines = 2, case["records"]
    elif k == "batch":
        stars, lines = case["stars"], int(1.03e5 * case["scale"])     # mean of exp U[ln 2e4, ln 3e5]
    grad = k not in FORWARD
    near = min(2 * case.get("W", 1500) + 1, int(2 * 20 * 1.9e5 / 2.998e10 * R) + 1)
    cells, pairs = stars * n * nd, stars * lines * nd
    flops = pairs * (near * (130 if grad else 40) + 40) + cells * (170 if grad else 112)
    if k == "scatter_step":
        flops += n * 2 * (nd ** 3 * 2 + nd * nd * 40) * 2
    bytes_ = cells * (24 + 4 + (4 if grad else 0)) + stars * lines * (48 + (8 if grad else 0)) + stars * n * 16
    return {"bytes": float(bytes_), "flops": float(flops)}


def tolerance(case):
    # 2-norm errors against the FP64 computation, measured over the listed and drawn cases:
    # opacity 2.3e-7, flux and f 3e-8 (both forms return the opacity and f in 32 bits);
    # gradients 2e-7, 3e-6 where a few lines dominate.  About four times that, and forty times
    # for the largest single difference against the output's rms.
    if case["kind"] == "solar_fp64":
        return {"rel": 1e-7, "max": 4e-6}
    if case["kind"] in FORWARD:
        return {"rel": 1e-6, "max": 4e-5}
    return {"rel": 1.2e-5, "max": 4e-4}


# ---------------------------------------------------------------------------------------------
# the same outputs in FP64
# ---------------------------------------------------------------------------------------------
_H, _KB, _C = 6.62607015e-27, 1.380649e-16, 2.99792458e10
_E, _ME, _EV, _AMU = 4.80320471e-10, 9.1093837015e-28, 1.602176634e-12, 1.66053906660e-24
_SQPI = math.sqrt(math.pi)
_EXACT_MOST = 4.0e9           # (line, point, layer) evaluations that exact() takes on


def _weideman(N=64):
    L = math.sqrt(N / math.sqrt(2.0))
    M = 4 * N
    th = math.pi * (np.arange(2 * M) - M + 0.5) / M
    t = L * np.tan(0.5 * th)
    psi = (L * L + t * t) * np.exp(-t * t)
    return np.array([np.mean(psi * np.cos(n * th)) for n in range(N + 1)]), L


def _voigt(v, a, want_d):
    """H(a, v) = Re w(v + i a) and dH/da: the Laplace series for |z| >= 8 (12 terms), Weideman's
    rational (order 64) inside."""
    v, a = torch.broadcast_tensors(v, a)
    z = torch.complex(v, a)
    q = 1.0 / z
    q2 = q * q
    c = [1.0]
    for n in range(12):
        c.append(c[-1] * (2 * n + 1) / 2.0)
    s = torch.full_like(z, c[12])
    for n in range(11, -1, -1):
        s = s * q2 + c[n]
    H = -(s * q).imag / _SQPI
    dH = None
    if want_d:
        s = torch.full_like(z, c[12] * 25)
        for n in range(11, -1, -1):
            s = s * q2 + c[n] * (2 * n + 1)
        dH = (s * q2).real / _SQPI
    near = (v * v + a * a) < 64.0
    if bool(near.any()):
        zn = z[near]
        coef, L = _weideman()
        iz = torch.complex(-zn.imag, zn.real)
        Z = (L + iz) / (L - iz)
        p = torch.full_like(zn, coef[64])
        for n in range(63, 0, -1):
            p = p * Z + coef[n]
        w = 2.0 * p / (L - iz) ** 2 + (1.0 / _SQPI) / (L - iz)
        H = H.clone()
        H[near] = w.real
        if want_d:
            dH = dH.clone()
            dH[near] = 2.0 * (zn.real * w.imag + zn.imag * w.real) - 2.0 / _SQPI
    return H, dH


def _expn(n, x):
    """E_n(x), n >= 1, in FP64: series for x <= 2, continued fraction above; E_n(0) = 1/(n - 1)."""
    ex = torch.exp(-x)
    xs = torch.clamp(x, 1e-300, 2.0)
    term, s = torch.ones_like(xs), torch.zeros_like(xs)
    for k in range(1, 40):
        term = term * (-xs / k)
        s = s + term / k
    e = -0.57721566490153286061 - torch.log(xs) - s
    for m in range(1, n):
        e = (torch.exp(-xs) - xs * e) / m
    xl = torch.clamp(x, min=2.0)
    f = xl + n + 2.0 * 60
    for k in range(60, 0, -1):
        f = xl + n + 2.0 * (k - 1) - k * (n - 1.0 + k) / f
    return torch.where(x <= 2.0, e, ex / f)


class _En(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x, n):
        ctx.save_for_backward(x)
        ctx.n = n
        return _expn(n, x)

    @staticmethod
    def backward(ctx, g):
        (x,) = ctx.saved_tensors
        return -g * _expn(ctx.n - 1, x), None


def _slab_integral(tau, S):
    """Int_0^tau_bottom S E_2 dt, S linear between layers and extrapolated to tau = 0."""
    s0 = (S[1] - S[0]) / (tau[1] - tau[0])
    t = torch.cat([torch.zeros_like(tau[:1]), tau])
    Sx = torch.cat([(S[0] - s0 * tau[0])[None], S])
    e3, e4 = _En.apply(t, 3), _En.apply(t, 4)
    D = t[1:] - t[:-1]
    sl = (Sx[1:] - Sx[:-1]) / D
    return (Sx[:-1] * (e3[:-1] - e3[1:]) + sl * (e4[:-1] - e4[1:] - D * e3[1:])).sum(0)


def _lambda_matrix(tau):
    """Rows of J = Lambda S [points][layer][layer]: the kernel E_1 / 2 against the hat function
    of each layer, from the second antiderivative E_3 of E_1; nothing below the bottom layer,
    the first segment extrapolated to tau = 0."""
    t = tau.transpose(0, 1)                                  # [points][nd]
    nd = t.shape[1]
    node = torch.cat([torch.zeros_like(t[:, :1]), t], 1)     # the top at 0, then the layers
    x = node[:, None, :] - t[:, :, None]                     # [points][row][node]
    ax = x.abs()
    e2, e3 = _En.apply(ax, 2), _En.apply(ax, 3)
    g1 = -torch.sign(x) * e2 / 2 + torch.sign(x) / 2         # first antiderivative of E_1(|x|)/2, 0 at x = 0
    g2 = e3 / 2 + ax / 2                                     # its antiderivative
    D = (node[:, 1:] - node[:, :-1])[:, None, :]
    one = g1[:, :, 1:] - g1[:, :, :-1]                       # Int k over a segment
    lin = g1[:, :, 1:] - (g2[:, :, 1:] - g2[:, :, :-1]) / D  # Int k (t - t_a)/D
    wa, wb = one - lin, lin
    lam = torch.zeros_like(x[:, :, 1:])
    lam[:, :, 0] += wb[:, :, 0] + wa[:, :, 1]
    lam[:, :, 1:-1] += wb[:, :, 1:-1] + wa[:, :, 2:]
    lam[:, :, -1] += wb[:, :, -1]
    r = (t[:, 0] / (t[:, 1] - t[:, 0]))[:, None]             # S(0) = S_0 (1 + r) - S_1 r
    lam[:, :, 0] += wa[:, :, 0] * (1 + r)
    lam[:, :, 1] -= wa[:, :, 0] * r
    return lam


def _flux(kappa, kc, sig, m, S_planck):
    """2 pi Int S E_2 dtau of one branch."""
    chi = kc + kappa + (0.0 if sig is None else sig)
    dm = (m[1:] - m[:-1])[:, None]
    tau = torch.cumsum(torch.cat([(chi[0] * m[0])[None], 0.5 * (chi[1:] + chi[:-1]) * dm]), 0)
    if sig is None:
        return 2 * math.pi * _slab_integral(tau, S_planck)
    out = []
    for a in range(0, tau.shape[1], 512):
        ta, Bp = tau[:, a:a + 512], S_planck[:, a:a + 512]
        eps = 1.0 - sig[:, a:a + 512] / chi[:, a:a + 512]
        lam = _lambda_matrix(ta)
        e = eps.transpose(0, 1)
        M = torch.eye(ta.shape[0], dtype=ta.dtype, device=ta.device) - (1.0 - e)[:, :, None] * lam
        S = torch.linalg.solve(M, (e * Bp.transpose(0, 1))[:, :, None])[:, :, 0]
        out.append(2 * math.pi * _slab_integral(ta, S.transpose(0, 1)))
    return torch.cat(out)


class _Star:
    """FP64 line data of one star on the torch device."""

    def __init__(self, at, grid, lines, corr, eos, dev):
        t = lambda x: torch.as_tensor(np.asarray(x, np.float64), device=dev)  # noqa: E731
        self.dev, self.n, self.W = dev, grid.n_lambda, lines.half_window
        self.lnr = math.log1p(1.0 / grid.R_grid)
        dgf, dg6, dab = corr if corr is not None else (np.zeros(lines.n_lines), np.zeros(lines.n_lines), None)
        x = np.log(lines.lambda_nm / grid.lambda0_nm) / self.lnr
        il = np.floor(x + 0.5)
        keep = (il >= -self.W) & (il <= self.n - 1 + self.W)
        self.keep = np.nonzero(keep)[0]
        sp = lines.species[keep]
        self.x, self.il = t(x[keep]), torch.as_tensor(il[keep].astype(np.int64), device=dev)
        T, rho = t(at.T), t(at.rho)
        mass = t(at.mass_amu)
        dv = torch.sqrt(2 * _KB * T[None] / (mass[:, None] * _AMU) + at.xi_cms ** 2)      # [ns][nd]
        pop = t(at.pop)
        if dab is not None:
            pop = pop * t(10.0 ** np.asarray(dab, np.float64)[eos])[:, None]
        s = torch.as_tensor(sp.astype(np.int64), device=dev)
        lc = t(lines.lambda_nm[keep] * 1e-7)[:, None]
        gf = t(10.0 ** (lines.log_gf[keep].astype(np.float64) + dgf[keep]))[:, None]
        E = t(lines.E_low_eV[keep])[:, None]
        idn = lc / dv[s]
        self.k = _C / dv[s]                                                               # [nl][nd]
        self.A = (math.pi * _E * _E / (_ME * _C)) / _SQPI * gf * (pop / rho)[s] * torch.exp(-E * _EV / (_KB * T)) * idn
        g6 = t(10.0 ** (lines.log_gamma6[keep].astype(np.float64) + dg6[keep]))[:, None] * t(at.n_pert)
        gr = t(10.0 ** lines.log_gamma_rad[keep].astype(np.float64))[:, None]
        g4 = t(10.0 ** lines.log_gamma4[keep].astype(np.float64))[:, None] * t(at.n_e)
        self.a = (gr + g4 + g6) * idn / (4 * math.pi)
        self.a6 = g6 * idn / (4 * math.pi)
        lam = grid.lambda0_nm * 1e-7 * torch.exp(torch.arange(self.n, device=dev, dtype=torch.float64) * self.lnr)
        self.stim = -torch.expm1(-_H * _C / _KB / (lam[None] * T[:, None]))
        self.B = 2 * _H * _C ** 2 / lam[None] ** 5 / torch.expm1(_H * _C / _KB / (lam[None] * T[:, None])) * 1e-7
        self.m = t(at.m)
        self.sp = sp

    def _chunks(self):
        step = max(1, int(6e6 // (2 * self.W + 1)))
        off = torch.arange(-self.W, self.W + 1, device=self.dev)
        for a in range(0, self.x.numel(), step):
            i = self.il[a:a + step, None] + off
            ok = (i >= 0) & (i < self.n)
            u = torch.expm1((self.x[a:a + step, None] - i) * self.lnr)
            yield slice(a, a + step), i.clamp(0, self.n - 1), ok, u

    def kappa(self):
        nd = self.k.shape[1]
        out = torch.zeros((nd, self.n), dtype=torch.float64, device=self.dev)
        for sl, i, ok, u in self._chunks():
            for d in range(nd):
                H, _ = _voigt(u * self.k[sl, d, None], self.a[sl, d, None], False)
                out[d].index_add_(0, i.reshape(-1), torch.where(ok, H * self.A[sl, d, None], 0.0).reshape(-1))
        return out * self.stim

    def line_sums(self, G):
        """(dL/dlog gf, dL/dlog gamma_6) of the star's lines from G = dL/dkappa [nd][n]."""
        nd = self.k.shape[1]
        Gs = G * self.stim
        g1, g2 = torch.zeros_like(self.x), torch.zeros_like(self.x)
        for sl, i, ok, u in self._chunks():
            for d in range(nd):
                H, dH = _voigt(u * self.k[sl, d, None], self.a[sl, d, None], True)
                gi = torch.where(ok, Gs[d][i], 0.0)
                g1[sl] += self.A[sl, d] * (gi * H).sum(1)
                g2[sl] += self.A[sl, d] * self.a6[sl, d] * (gi * dH).sum(1)
        return math.log(10.0) * g1, math.log(10.0) * g2


def _inst_matrix(inst, grid, dev):
    """Dense rows of the instrument: shift, broadening and LSF as one Gaussian in ln lambda."""
    lnr = math.log1p(1.0 / grid.R_grid)
    sl = 1.0 / (2 * math.sqrt(2 * math.log(2.0)) * inst.R_lsf)
    sig = math.sqrt(sl ** 2 + (inst.v_b_kms * 1e5 / _C) ** 2) / lnr
    cp = np.log(inst.pix_lambda_nm / (1 + inst.v_r_kms * 1e5 / _C) / grid.lambda0_nm) / lnr
    i0, i1 = np.ceil(cp - 5 * sig).astype(int), np.floor(cp + 5 * sig).astype(int)
    K = np.zeros((cp.size, grid.n_lambda))
    for p in range(cp.size):
        i = np.arange(max(i0[p], 0), min(i1[p], grid.n_lambda - 1) + 1)
        g = np.exp(-0.5 * ((i - cp[p]) / sig) ** 2)
        K[p, i] = g / g.sum()
    return torch.as_tensor(K, device=dev)


def exact(case, seed):
    k = case["kind"]
    if k in ("joint", "group", "batch") or case.get("eta"):
        return None
    prob, _, y, w, corr = _host(case, seed)
    evals = prob.n_evals * (1 if k in FORWARD else 2)
    if evals > _EXACT_MOST or prob.grid.n_lambda > 9000:
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    fwd_only = k in FORWARD
    star = _Star(prob.atmos, prob.grid, prob.lines, None if fwd_only else corr, prob.elem_of_species, dev)
    t = lambda a: torch.as_tensor(np.asarray(a, np.float64), device=dev)  # noqa: E731
    kc, sig = t(prob.kappa_c), None if prob.sigma_c is None else t(prob.sigma_c)
    kap = star.kappa().requires_grad_(not fwd_only)
    F = _flux(kap, kc, sig, star.m, star.B)
    Fc = _flux(torch.zeros_like(kc), kc, sig, star.m, star.B)
    if prob.instrument is not None:
        K = _inst_matrix(prob.instrument, prob.grid, dev)
        f = (K @ F) / (K @ Fc)
    else:
        f = F / Fc
    if fwd_only:
        out = {"F": F.detach(), "Fc": Fc, "f": f.detach()}
        if k != "forward":
            out["kappa"] = kap.detach()
        return out
    r = t(y) - f
    loss = (t(w) * r * r).sum()
    G, = torch.autograd.grad(loss, kap)
    s1, s2 = star.line_sums(G)
    nl = prob.lines.n_lines
    g_gf, g_g6 = torch.zeros(nl, dtype=torch.float64, device=dev), torch.zeros(nl, dtype=torch.float64, device=dev)
    idx = torch.as_tensor(star.keep, device=dev)
    g_gf[idx], g_g6[idx] = s1, s2
    g_ab = torch.zeros(N_ELEM, dtype=torch.float64, device=dev)
    g_ab.index_add_(0, torch.as_tensor(prob.elem_of_species[star.sp].astype(np.int64), device=dev), s1)
    out = {"f": f.detach(), "loss": loss.detach() if k == "autograd" else loss.detach().reshape(1), "g_gf": g_gf,
           "g_g6": g_g6, "g_ab": g_ab}
    if k != "autograd":
        out["dL"] = (-2 * t(w) * r).detach()
    return out
