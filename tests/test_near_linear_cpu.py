"""The bound that the near-linear float sweep puts on what it leaves out, against the exact arc-length weights.

In units of second differences, with T_a, T_b the third differences of a stencil, u the middle of its central interval
and e = eps / dx^2, the sweep's deviations from the linear scheme are quadratic forms over u / (u^2 + 1 + e); the
bound's coefficients are read from the kernel's header.  Extended precision leaves ten digits of the smallest
omission drawn here.
"""
import os
import re

import numpy as np

from paper_1909_13263_gb300 import build

LD = np.longdouble


def _coefficients():
    text = open(os.path.join(build.CSRC, "alw_sweep32.cuh")).read()
    return [float(re.search(r"constexpr float %s = ([0-9.e-]+)f;" % n, text).group(1))
            for n in ("kNearT", "kNearTW", "kNearTWW")]


def _mean(a, b):
    """Mean of sqrt(1 + x^2) over [a, b] (2 |b - a| well below the size of the roots): sigma/2 - B(t^2)/sigma."""
    sigma = np.sqrt(1 + a * a) + np.sqrt(1 + b * b)
    x = ((b - a) / sigma) ** 2
    c = np.zeros_like(x)
    for k in range(30, 0, -1):
        c = c * x + LD(2 * k) / LD(2 * k + 1)
    return sigma / 2 - c * x / sigma


def _exact(d1, d2, d3, d4, e):
    """Deviations of phi^- and (the node before) phi^+ from the linear scheme, over dx."""
    q = [(e + _mean(a, b) ** 2) ** 2 for a, b in ((d2, 2 * d2 - d1), (d2, d3), (2 * d3 - d4, d3))]
    ta, tb = d1 - 2 * d2 + d3, d2 - 2 * d3 + d4
    lin = [LD(1) / 10, LD(6) / 10, LD(3) / 10]

    def weights(p):
        w = [g / x for g, x in zip(lin, p)]
        return w[0] / sum(w) - lin[0], w[2] / sum(w) - lin[2]

    m0, m2 = weights(q)
    p0, p2 = weights(q[::-1])
    return -(m0 * 2 * ta + m2 * tb) / 6, (p0 * 2 * tb + p2 * ta) / 6


def test_bound_covers_what_the_near_linear_form_leaves_out():
    kt, ktw, ktww = _coefficients()
    rng = np.random.default_rng(11)
    n = 400000

    def size(lo, hi):
        return (10 ** rng.uniform(lo, hi, n) * rng.choice([-1, 1], n)).astype(LD)

    t, w, u = size(-6, -0.5), size(-4, 0), size(-3, 2)
    e = np.where(rng.random(n) < 0.5, 0, 10 ** rng.uniform(-6, 2, n)).astype(LD)
    ta, tb = t, t * rng.uniform(-1, 1, n).astype(LD)
    swap = rng.random(n) < 0.5
    ta, tb = np.where(swap, tb, ta), np.where(swap, ta, tb)
    d2, d3 = u, u + w
    d1, d4 = d2 - (w - ta), d3 + (w + tb)
    minus, plus = _exact(d1, d2, d3, d4, e)
    y = u + w / 2
    k = y / (y * y + 1 + e) / 100
    left = np.maximum(np.abs(minus + k * (6 * ta * ta - 3 * ta * tb + 7 * tb * tb)),
                      np.abs(plus - k * (7 * ta * ta - 3 * ta * tb + 6 * tb * tb)))
    tm = np.maximum(np.abs(ta), np.abs(tb))
    wm = np.maximum(np.abs(w), np.maximum(np.abs(w - ta), np.abs(w + tb)))
    assert (left / (tm * tm * (kt * tm + ktw * wm + ktww * wm * wm))).max() <= 1
