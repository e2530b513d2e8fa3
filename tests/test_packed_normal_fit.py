"""Where the polynomials of the packed Box-Muller transform (zo_device.cuh: box_muller_parts) come
from: minimax fits to the functions themselves, by Lawson's iteratively reweighted least squares
(C. L. Lawson, Contributions to the theory of linear least maximum approximation, 1961) in
extended precision, with the committed coefficients' errors against the functions.

With x = m - 1, m in [2/3, 4/3):    -2 ln(1 + x) = -2 x + x^2 R(x),  g = 2 x,  P(g) = -R(x) / 4
with v = t^2, t in [-1, 1]:          sin(pi/4 t) = t (s0 + q(v)),     s0 = fp32(pi/4)
                                     cos(pi/4 t) = 1 + v p(v)
"""

import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LD = np.longdouble
QUARTER_PI = LD("0.785398163397448309615660845819875721")


def committed(name):
    """The coefficients of the constant array `name`, lowest order first."""
    path = os.path.join(ROOT, "paper_2608_15665_gb300", "csrc", "zo_device.cuh")
    text = re.search(r"constexpr float %s\[\d+\] = \{([^}]*)\}" % name, open(path, encoding="utf-8").read())
    return [float.fromhex(c.strip().rstrip("f")) for c in text.group(1).split(",")]


def minimax(F, x, orders, w, steps=400):
    """Coefficients c of x^j, j in orders, that minimise max w |F - sum c x^j| over the points x."""
    A = np.stack([x**j for j in orders], 1)
    A = A / (scale := np.abs(A).max(axis=0))
    lam, best = np.ones(len(x), dtype=LD) / len(x), None
    for _ in range(steps):
        s = np.sqrt(lam) * w
        M = A * s[:, None]
        c = np.linalg.lstsq(M.astype(np.float64), (F * s).astype(np.float64), rcond=None)[0].astype(LD)
        rest = (F * s - M @ c).astype(np.float64)       # one refinement: the solver is in 64 bits
        c = c + np.linalg.lstsq(M.astype(np.float64), rest, rcond=None)[0]
        e = np.abs((F - A @ c) * w)
        if best is None or e.max() < best[0]:
            best = e.max(), c / scale
        lam = lam * (e + LD(1e-30))
        lam /= lam.sum()
    return best[1]


def points(lo, hi, n=600):
    t = np.cos(np.pi * (np.arange(n, dtype=LD) + 0.5) / n)
    return (lo + hi) / 2 + (hi - lo) / 2 * t


def log_case():
    x = points(LD(2) / 3 - 1, LD(4) / 3 - 1)
    want = [-c * 4 * 2.0**k for k, c in enumerate(committed("kP"))]      # of R
    return x, (-2 * np.log1p(x) + 2 * x) / x**2, np.abs(x) / 2, want


def sin_case():
    v = points(LD(0), LD(1))
    s0 = LD(float(np.float32(float(QUARTER_PI))))
    return v, np.sin(QUARTER_PI * np.sqrt(v)) / np.sqrt(v) - s0, np.ones_like(v), committed("kS")


def cos_case():
    v = points(LD(0), LD(1))
    F = (np.cos(QUARTER_PI * np.sqrt(v)) - 1) / v
    return v, F, np.maximum(v, LD("0.05")), committed("kC")


@pytest.mark.parametrize("case, fixed", [(log_case, {0: 1.0}), (sin_case, {})])
def test_fits_rounded_from_the_lowest_order_on(case, fixed):
    """ln (relative error, R(0) = 1 given) and sin: a coefficient is rounded to fp32, lowest order
    first, and the rest are fitted again."""
    x, F, w, want = case()
    for j, c in enumerate(want):
        assert float(np.float32(c)) == c
        if j in fixed:
            assert c == fixed[j]
            continue
        left = F - sum(LD(a) * x**k for k, a in enumerate(want[:j]))
        got = minimax(left, x, range(j, len(want)), w)[0]
        # the fit in other arithmetic may round to a neighbour
        assert abs(float(got) - c) <= 2.0**-23 * abs(c), (j, float(got).hex(), c.hex())


def test_cos_fit_rounded_at_once():
    v, F, w, want = cos_case()
    for got, c in zip(minimax(F, v, range(4), w), want):
        assert abs(float(got) - c) <= 2.0**-21 * abs(c), (float(got).hex(), c.hex())


def test_errors_of_the_committed_polynomials():
    """In exact arithmetic: ln 5.8e-9 of the result, sin 2.5e-9, cos 8.7e-9 (the rounding of its
    first coefficient); all below half a unit in the last place of fp32 results near 1, 3e-8."""
    x, _, _, R = log_case()
    ln = -2 * np.log1p(x)
    e = np.abs(-2 * x + x**2 * sum(LD(c) * x**k for k, c in enumerate(R)) - ln) / np.abs(ln)
    assert 5.0e-9 < e.max() <= 5.9e-9
    t = points(LD(-1), LD(1))
    v, s0 = t * t, LD(float(np.float32(float(QUARTER_PI))))
    s = t * (s0 + sum(LD(c) * v**k for k, c in enumerate(committed("kS"))))
    assert np.abs(s - np.sin(QUARTER_PI * t)).max() <= 2.5e-9
    c = 1 + v * sum(LD(a) * v**k for k, a in enumerate(committed("kC")))
    assert np.abs(c - np.cos(QUARTER_PI * t)).max() <= 8.7e-9
