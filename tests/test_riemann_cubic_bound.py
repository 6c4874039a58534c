"""The bound behind the stopping rule of the kernels' FP64 star-velocity iteration (Sec. 2.1 flux).

The iteration u <- u - d (1 + d phi''/(2 phi')), d = phi/phi', on phi(u) = p_1(u) - p_3(u) ends once
|d| <= 3e-6 c. The error left is C3 |d|^3 with C3 = |phi''^2/(2 phi'^2) - phi'''/(6 phi')| at the root;
C3 c^2 < 2 makes it less than 6e-17 c. Checked in 40-digit arithmetic on seeded states with |u| up to
100 c, with the wave curves restated from the PDE; and that one step from an error of 3e-6 c ends there.
"""
import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
from test_riemann_newton_bound import wave1, wave3  # noqa: E402


def test_cubic_constant_below_bound():
    mp.mp.dps = 40
    rng = np.random.default_rng(41)
    worst, worst_step = 0.0, 0.0
    for R in (0.05, 0.5, 4.0, 20.0, 100.0):
        for _ in range(24):
            ul, ur = [mp.mpf(x) for x in rng.uniform(-R, R, 2)]
            pl, pr = [mp.mpf(x) for x in rng.uniform(-R * R, R * R, 2)]
            phi = lambda u: wave1(u, ul, pl, mp.mpf(1)) - wave3(u, ur, pr, mp.mpf(1))
            lo, hi = -mp.mpf(10 * R * R + 10), mp.mpf(10 * R * R + 10)
            for _ in range(150):
                mid = (lo + hi) / 2
                lo, hi = (mid, hi) if phi(mid) > 0 else (lo, mid)
            r = (lo + hi) / 2
            d1, d2, d3 = [mp.diff(phi, r, n) for n in (1, 2, 3)]
            worst = max(worst, float(abs(d2 * d2 / (2 * d1 * d1) - d3 / (6 * d1))))
            u = r + mp.mpf("3e-6")
            f, g, h = phi(u), mp.diff(phi, u, 1), mp.diff(phi, u, 2)
            d = f / g
            worst_step = max(worst_step, float(abs(u - d * (1 + d * h / (2 * g)) - r)))
    assert worst < 2.0, worst
    assert worst_step < 6e-17, worst_step
