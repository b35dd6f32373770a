"""The polynomials of box_muller_t (csrc/lb_collide.cuh): where they come from and how far off they are, in 64
bits.  Each is the weighted minimax polynomial of its degree, found by Lawson's iteration (least squares,
reweighted by the residual) on Chebyshev nodes of its interval."""
import os
import re

import numpy as np
import pytest

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0710_1272_gb300", "csrc",
                      "lb_collide.cuh")


def _lawson(fn, weight, a, b, degree, turns=120):
    n = 4000
    x = (a + b) / 2 + (b - a) / 2 * np.cos(np.pi * (np.arange(n) + 0.5) / n)
    y, wt, w = fn(x), weight(x), np.ones(n)
    powers = np.vander(x, degree + 1, increasing=True)
    for _ in range(turns):
        s = np.sqrt(w) * wt
        c = np.linalg.lstsq(powers * s[:, None], y * s, rcond=None)[0]
        r = np.abs((powers @ c - y) * wt)
        w *= r / r.max() + 1e-3
        w /= w.sum()
    return r.max(), x, y, wt


def _coefficients():
    """Those of the source, highest power first: logarithm, sine, cosine."""
    text = open(HEADER).read()
    body = text[text.index("box_muller_t(typename O::V u1"):]
    body = body[:body.index("n1 = O::mul(rad")]
    num = r"splat\((-?[\d.]+(?:e-?\d+)?)f\)"
    log = [float(v) for v in re.findall(num, body[body.index("V q = "):body.index("q = O::mul(f")])]
    sine = [float(v) for v in re.findall(num, body[body.index("V s = "):body.index("// the leading")])]
    lead = [float(v) for v in re.findall(num, body[body.index("// the leading"):body.index("V c = ")])]
    cosine = [float(v) for v in re.findall(num, body[body.index("V c = "):body.index("float k[O::N]")])]
    return log, sine + [sum(lead)], cosine


def _log_q(f):
    f = np.where(np.abs(f) < 1e-3, 1e-3, f)
    return (np.log1p(f) - f + f * f / 2) / f**3


# name, function, weight, interval, degree, error stated in the source
FITS = [
    # ln(1 + f) = f - f^2/2 + f^3 Q(f), error relative to the logarithm
    ("log", _log_q, lambda f: np.abs(f**3 / np.log1p(np.where(f == 0, 1e-9, f))), 0.5**0.5 - 1, 2**0.5 - 1, 7, 6e-9),
    # sin(pi r) = r S(r^2), relative to pi r
    ("sine", lambda t: np.sin(np.pi * np.sqrt(t)) / np.sqrt(t), lambda t: 1 / np.pi + 0 * t, 1e-9, 1 / 16, 3, 3.1e-9),
    # cos(pi r) = 1 + r^2 C(r^2), absolute
    ("cosine", lambda t: (np.cos(np.pi * np.sqrt(t)) - 1) / t, lambda t: t, 1e-9, 1 / 16, 3, 6e-11),
]


@pytest.mark.parametrize("k", range(3))
def test_polynomial(k):
    name, fn, weight, a, b, degree, stated = FITS[k]
    c = _coefficients()[k]
    if name == "cosine":
        assert c.pop() == 1.0
    assert len(c) == degree + 1
    best, x, y, wt = _lawson(fn, weight, a, b, degree)
    off = np.abs(np.polyval(c, x) - y) * wt
    # the coefficients are rounded to single precision: half an ulp of each, at its power's largest
    largest = max(abs(a), abs(b))
    rounding = sum(2.0**-25 * 2 * abs(v) * largest**p for p, v in enumerate(reversed(c)))
    print(name, "largest error %.2e, of the fit %.2e" % (off.max(), best))
    assert best <= stated
    assert off.max() <= best + (wt * rounding).max()
