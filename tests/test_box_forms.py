"""CPU pins of the box expansions of the far wings, in FP64 NumPy: the truncated Chebyshev
expansion of f(D) = (eps/u)^2 over two boxes, the derivative operators that turn it into
f^2..f^4, and the few moments kept at the windows' ends."""
import math
import os
import re

import numpy as np
import pytest


def order(o):
    """The kernels' expansion order at box offset o (box_order)."""
    for lim, p in ((90, 3), (33, 4), (19, 5), (14, 6), (9, 7), (7, 8), (6, 9), (5, 10), (4, 11)):
        if o >= lim:
            return p
    return 13


def coefficients(o, B, L, N=16):
    h = B / 2
    th = np.pi * (np.arange(N) + 0.5) / N
    X = np.cos(th)
    f = (L * h / np.expm1((o * B + h * (X[:, None] - X[None, :])) * L)) ** 2
    T = np.cos(np.outer(np.arange(N), th)) * 2 / N
    T[0] /= 2
    C = T @ f @ T.T
    k = np.arange(N)
    C[k[:, None] + k[None, :] > order(abs(o))] = 0.0
    return C[:14, :14]


def operators(eps, P=13):
    D = np.zeros((P + 1, P + 1))
    for k in range(1, P + 1):
        d = np.polynomial.chebyshev.chebder(np.eye(P + 1)[k])
        D[:d.size, k] = d
    A = [np.eye(P + 1)]
    for q, m in enumerate((6.0, 20.0, 42.0)):
        A.append((D + (2 * q + 3) * eps * np.eye(P + 1)) @ (D + (2 * q + 2) * eps * np.eye(P + 1)) @ A[-1] / m)
    return A


def series(a):
    """beta_n and gamma_n: H sqrt(pi)/(A a) and dH/da sqrt(pi)/A as series in p = 1/v^2."""
    s = a * a
    return ((1, 1.5 - s, 3.75 - 5 * s + s ** 2, 13.125 - 26.25 * s + 10.5 * s ** 2 - s ** 3),
            (1, 1.5 - 3 * s, 3.75 - 15 * s + 5 * s ** 2, 13.125 - 78.75 * s + 52.5 * s ** 2 - 7 * s ** 3))


@pytest.mark.parametrize("B,L", [(32, 3.33e-6), (16, 1e-5), (4, 1e-4)])
@pytest.mark.parametrize("o", [3, 4, 5, 6, 7, 9, 14, 19, 33, 45, 90])
def test_expansion_of_all_four_terms(B, L, o):
    # |v| = 20 at the nearest distance any class allows (two boxes), damping up to v/9
    h = B / 2
    eps = L * h
    x = np.linspace(-1, 1, 41)
    T = np.polynomial.chebyshev.chebvander(x, 13)
    A = operators(eps)
    kap = (math.expm1(2 * B * L) / eps) ** 2 / 400
    for s in (1, -1):
        C = coefficients(s * o, B, L)
        p = kap * (eps / np.expm1((s * o * B + h * (x[:, None] - x[None, :])) * L)) ** 2
        for a in (0.0, 0.6, 2.2):
            for w in series(a):
                got = sum(w[q] * kap ** (q + 1) * (T @ A[q]) for q in range(4)) @ C @ T.T
                ref = p * (w[0] + p * (w[1] + p * (w[2] + p * w[3])))
                err = np.abs(got / ref - 1)
                assert err.max() < (1.0e-7 if o == 3 else 4e-8)      # measured 9.3e-8, 3.5e-8: at the corners
                assert np.sqrt(np.mean(err ** 2)) < 1.5e-8           # over the two boxes


@pytest.mark.parametrize("cls", [0, 1, 2, 3])
def test_series_against_faddeeva(cls):
    """The four terms at the distances of a separation class, |v| >= 20 2^cls with damping up to |v|/9.  The first
    dropped term of H is (a/v)^8 = 2.3e-8 there, that of dH/da nine times that."""
    wofz = pytest.importorskip("scipy.special").wofz
    v = np.geomspace(20.0 * 2 ** cls, 400.0 * 2 ** cls, 400)[None, :]
    a = np.geomspace(1e-3, 20.0 * 2 ** cls / 9, 60)[:, None]
    p = 1 / v ** 2
    w = wofz(v + 1j * a)
    H, dH = w.real, 2 * (v * w.imag + a * w.real) - 2 / math.sqrt(math.pi)
    for n, (ref, f) in enumerate(((H, a), (dH, 1.0))):
        c = series(a)[n]
        got = f * p * (c[0] + p * (c[1] + p * (c[2] + p * c[3]))) / math.sqrt(math.pi)
        # the reference's dH/da is a difference of numbers near 1: 2e-16 / dH/da
        tol = 2.4e-8 if n == 0 else 2.2e-7 + 4e-16 / np.abs(ref)
        err = np.abs(got / ref - 1)
        print("class %d, %s: %.2e" % (cls, "dH/da" if n else "H", np.max(err - (tol - 2.2e-7 if n else 0.0))))
        assert np.all(err < tol)


@pytest.mark.parametrize("W,B,L", [(1500, 32, 3.33e-6), (2000, 32, 3.33e-6), (287, 32, 3.33e-6), (67, 4, 1e-4)])
def test_window_ends_with_few_moments(W, B, L):
    omax = (W + 1) // B - 1
    KE = 5 if order(omax + 1) <= 4 else 8
    h = B / 2
    x = np.linspace(-1, 1, 41)
    T = np.polynomial.chebyshev.chebvander(x, 13)
    for e in (1, 2):
        for s in (1, -1):
            C = coefficients(s * (omax + e), B, L)
            f = (L * h / np.expm1((s * (omax + e) * B + h * (x[:, None] - x[None, :])) * L)) ** 2
            assert np.all(C[KE:] == 0.0)
            assert np.abs(T[:, :KE] @ C[:KE] @ T.T / f - 1).max() < 4e-8


def coefficient(n, k):
    """(-1)^k c_(n-k) binom(2n + 1, 2k + 1), c_m = (2m - 1)!!/2^m."""
    c = 1.0
    for m in range(n - k):
        c *= (2 * m + 1) / 2.0
    return (-1) ** k * c * math.comb(2 * n + 1, 2 * k + 1)


@pytest.mark.parametrize("terms,vmin,a_max,tol_h,tol_d", [
    (8, 6.0, math.sqrt(1.5), 6.4e-8, 1.3e-7), (4, 20.0, math.sqrt(1.5), 3e-9, 2e-8), (3, 30.0, math.sqrt(1.5), 2.7e-8, 4.7e-8),
    (8, 20.0, math.sqrt(44.0), 3.7e-9, 7.2e-8)])
def test_series_of_the_nearer_cells(terms, vmin, a_max, tol_h, tol_d):
    """The far-wing kernels' series at the smallest |v| each form takes and up to its largest damping (a^2 <= 1.5, the
    wide form a^2 <= 44): H relative, dH/da against its scale p/sqrt(pi) (it crosses zero)."""
    wofz = pytest.importorskip("scipy.special").wofz
    v = np.concatenate([np.linspace(vmin, 4 * vmin, 600)])[None, :]
    a = np.concatenate([np.geomspace(1e-3, 1.0, 25), np.linspace(1.0, a_max, 40)])[:, None]
    w = wofz(v + 1j * a)
    H, dH = w.real, 2 * (v * w.imag + a * w.real) - 2 / math.sqrt(math.pi)
    p, s = 1 / v ** 2, a * a
    got_h = got_d = 0.0
    for n in range(terms):
        got_h = got_h + p ** (n + 1) * sum(coefficient(n, k) * s ** k for k in range(n + 1))
        got_d = got_d + p ** (n + 1) * sum((2 * k + 1) * coefficient(n, k) * s ** k for k in range(n + 1))
    assert np.max(np.abs(got_h * a / math.sqrt(math.pi) / H - 1)) < tol_h
    # the reference's dH/da is a difference of numbers near 1 at 2e-16 each
    assert np.max(np.abs(got_d / math.sqrt(math.pi) - dH) / (p / math.sqrt(math.pi)) - 1e-15 * v ** 2) < tol_d


def test_coefficients_of_the_source():
    """The far-wing kernels' coefficients as they stand in the source are those of the series above, every power of
    a^2 up to a^14 included."""
    path = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_24141_gb300", "csrc",
                        "pz_far.cuh")
    with open(path) as f:
        body = f.read().split("void poly_coeffs(")[1].split("#undef PZ_Q")[0]
    parts = re.split(r"c\[(\d)\] = ", body)
    assert [int(n) for n in parts[1::2]] == list(range(8)) and not re.findall(r"PZ_Q\(\d", parts[2])
    for n, text in zip(range(1, 8), parts[4::2]):
        got = {int(k): float(v) for k, v in re.findall(r"PZ_Q\((\d), (-?[\d.]+)f\)", text)}
        assert got == {k: coefficient(n, k) for k in range(n + 1)}
