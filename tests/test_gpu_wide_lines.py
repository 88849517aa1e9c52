"""Very wide lines (fast microturbulence, light species in hot gas): the mixed form against the plain
FP64 form.  The series of the far wings hold K^8, K = 4^uexp/k^2 with k = c/dv_D, which has to stay
inside FP32 whatever the lines' width."""
import numpy as np
import pytest

import paper_2607_24141_gb300 as pz
from paper_2607_24141_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def problem(xi_kms, teff, masses, mu, g4=0.0, n=1500, lines=600, W=1200, ns=8):
    at = I.make_atmosphere(teff, 4.0, ns, 5, log_abund_mean=mu, xi_kms=xi_kms)
    at.mass_amu[:] = np.geomspace(masses[0], masses[1], ns)
    grid = I.Grid(1600.0, 3e5, n)
    rng = np.random.default_rng(5)
    hi = float(I.grid_lambda_nm(grid)[-1])
    parts = list(I._atomic_lines(rng, lines, 1600.0 * (1 - W / 3e5), hi * (1 + W / 3e5), np.arange(ns)))
    parts[5] = parts[5] + g4
    return I.Problem("wide", at, grid, I._pack([tuple(parts)], W), I.make_kappa_c(at, grid))


def outputs(prob, prec):
    import torch
    s = pz.Synthesizer(prob, prec)
    kl = torch.empty((s.n_depth, s.n_lambda), dtype=torch.float32, device=s.device)
    f = s.forward(kl)
    dL = torch.tensor(np.random.default_rng(1).normal(size=tuple(f.shape)), dtype=torch.float32, device=s.device)
    g = [torch.empty(s.n_lines, dtype=torch.float32, device=s.device) for _ in range(4)]
    s.backward4(dL, *g)
    out = [t.double().cpu().numpy() for t in [kl, f] + g]
    s.close()
    return out


@pytest.mark.parametrize("xi,teff,masses,mu,g4", [
    (30.0, 4500.0, (12.0, 60.0), -10.0, 0.0),
    (100.0, 4500.0, (12.0, 60.0), -4.0, 0.0),       # K^8 above 2^103 at a fixed scale of 2^36
    (300.0, 6000.0, (12.0, 60.0), -6.0, 0.0),
    (1.0, 20000.0, (1.0, 4.0), -3.0, 2.0),          # strong, strongly damped lines of hydrogen and helium masses
    (0.0, 30000.0, (1.0, 238.0), -5.0, 1.0),        # K from 1 down to 1/238
    (0.0, 2500.0, (238.0, 238.0), -9.0, 0.0),       # narrow lines: k near 10^6
])
def test_wide_lines_against_the_plain_form(xi, teff, masses, mu, g4):
    prob = problem(xi, teff, masses, mu, g4)
    got, ref = outputs(prob, pz.PZ_MIXED), outputs(prob, pz.PZ_FP64)
    for a in got:
        assert np.all(np.isfinite(a))
    m = ref[0] > 0
    assert np.max(np.abs(got[0][m] / ref[0][m] - 1)) < 3e-5       # the mixed form's bar on kappa
    print("kappa, f, gradients:", ["%.1e" % (np.linalg.norm(a - b) / np.linalg.norm(b)) for a, b in zip(got, ref)])
    assert np.linalg.norm(got[0] - ref[0]) < 2e-6 * np.linalg.norm(ref[0])
    for a, b in zip(got[2:], ref[2:]):
        assert np.linalg.norm(a - b) < 1e-5 * np.linalg.norm(b)


def test_plain_form_with_unbounded_damping():
    """A damping whose square leaves FP64 gives the line no profile, not NaN (the plain FP64 form)."""
    prob = problem(1.0, 5000.0, (12.0, 60.0), -9.0, lines=300)
    none = problem(1.0, 5000.0, (12.0, 60.0), -9.0, lines=300)
    for k in (0, 7, 150):
        prob.lines.log_gamma_rad[k] = 200.0       # a near 10^187
        none.lines.log_gf[k] = -300.0             # the same lines without strength
    got, ref = outputs(prob, pz.PZ_FP64), outputs(none, pz.PZ_FP64)
    for a, b in zip(got[:2], ref[:2]):
        assert np.all(np.isfinite(a))
        assert np.array_equal(a, b)
    for a in got[2:]:
        assert np.all(np.isfinite(a))
