"""Fit the polynomial of the FP32 arc-cosine map on c in [0, 1].

J(c) = sqrt(1 - c^2) + c (pi - arccos c) = pi c + (1 - c)^{3/2} B(c), with B
analytic on [0, 1] (its nearest singularity is at c = -1; B(1) = 2 sqrt(2)/3).
B is approximated by a polynomial of degree ``DEG`` minimising the maximum
ABSOLUTE error of J (Lawson's iteratively re-weighted least squares on a dense
Chebyshev grid); targets are computed with 40-digit mpmath through
theta = arccos c, J - pi c = sin(theta) - theta cos(theta), to avoid the
cancellation near c = 1.  For c in [-1, 0) the map uses
J(c) = J(|c|) + pi min(c, 0).  Run ``python fit_jpos.py`` to print the table
that nk_map.cuh embeds, and ``python fit_jpos.py pi`` for nk_f32x2.cuh's: J / pi =
c + (1 - c)^{3/2} P(c), P = B / pi.

There the coefficients are FP32 numbers, rounded one after the other from the
constant on, each time with the others fitted again: rounding them all at the
end leaves errors of one sign, which a net of eight layers adds up.  The relative
error counts fully from c = 0.3 on, where the layers after the first have their
correlations (at c = 0 the constant 1 / pi alone is off by 4.0e-8), and is fitted
around -3e-9, against the bias of the same size that the FP32 evaluation has.
"""

import sys

import mpmath as mp
import numpy as np

DEG = 5
mp.mp.dps = 40


def target(c):
    c = mp.mpf(c)
    if c == 1:
        return 2 * mp.sqrt(2) / 3
    t = mp.acos(c)
    return (mp.sin(t) - t * mp.cos(t)) / (1 - c) ** mp.mpf(1.5)


def fit(deg=DEG, n=3000, iters=300):
    x = (np.cos(np.pi * (np.arange(n) + 0.5) / n) + 1) / 2
    B = np.array([float(target(v)) for v in x])
    wgt = (1 - x) ** 1.5
    V = np.vander(x, deg + 1, increasing=True)
    w = np.ones(n)
    for _ in range(iters):
        sw = np.sqrt(w) * wgt
        c, *_ = np.linalg.lstsq(V * sw[:, None], B * sw, rcond=None)
        err = np.abs((V @ c - B) * wgt)
        w = w * (err + 1e-30)
        w /= w.sum()
    return c


def fit_pi(deg=DEG, n=4000, iters=40, low=0.3, low_weight=0.02, bias=-3e-9):
    x = np.arange(n) / n
    w3 = (1 - x) ** 1.5
    T = np.array([float(target(v)) for v in x]) / np.pi
    J = x + w3 * T
    V = np.vander(x, deg + 1, increasing=True) * (w3 / J)[:, None]
    y = w3 * T / J + np.where(x > low, bias, 0.0)
    wt = np.where(x > low, 1.0, low_weight)

    def rest(fixed):
        k0 = len(fixed)
        r = y - V[:, :k0] @ np.array(fixed)
        w = wt.copy()
        for _ in range(iters):
            sw = np.sqrt(w)
            c, *_ = np.linalg.lstsq(V[:, k0:] * sw[:, None], r * sw, rcond=None)
            err = np.abs(V[:, k0:] @ c - r) * np.sqrt(wt)
            w = w * (err / err.mean() + 1e-3)
            w /= w.mean()
        return c, err.max()

    b = [float(np.float32(1 / np.pi))]
    for k in range(1, deg):
        v = np.float32(rest(b)[0][0])
        near = [v, np.nextafter(v, np.float32(1)), np.nextafter(v, np.float32(-1))]
        b.append(min((float(q) for q in near), key=lambda q: rest(b + [q])[1]))
    return b + [float(np.float32(rest(b)[0][0]))]


if __name__ == "__main__":
    if sys.argv[1:] == ["pi"]:
        for i, ci in enumerate(fit_pi()):
            print("  %.9e,  // c^%d" % (ci, i))
        sys.exit()
    c = fit()
    xs = np.linspace(0, 1, 20001)
    Jt = np.array([float(mp.pi * v + (1 - mp.mpf(v)) ** mp.mpf(1.5) * target(v)) for v in xs[::20]])
    Ja = np.pi * xs[::20] + (1 - xs[::20]) ** 1.5 * np.polyval(c[::-1], xs[::20])
    print("max abs err of J (float64 eval): %.3e" % np.abs(Ja - Jt).max())
    for i, ci in enumerate(c):
        print("  %.9e,  // c^%d" % (ci, i))
