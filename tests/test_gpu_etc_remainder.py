"""ETC's derivative through the tree's multipoles ends at rounding for a single dipole at the corner of its
leaf seen from the nearest point that takes the leaf's multipoles, where an expansion cut too early shows
first: against the directly summed derivative, at the smallest order that goes through the tree (20)."""
import math

import numpy as np
import pytest

from paper_1910_10863_gb300 import workloads as W
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu


def test_dipole_at_the_corner_of_its_leaf():
    """A small polygon about the root's centre, where four leaves meet; elements of 0.00196, so that all points
    and images lie at 54 to 790 lengths, where both sides take three nodes.  The remainder is 2e-16 of the dipole's
    derivative h / (2 pi r^2) and 21 steps of each recurrence round to 21 eps: 1e-14.  (With the cut at
    10^-14.7 it is 21 (s / r)^20, s the dipole's and r the point's distance from the leaf's centre: 5e-14.)"""
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    w = W.single_fiber(0.005, 16, 1.0, 1.2, 0.8, 0.3)
    s = pf.Solver(w, p=20, depth=3)
    plan = s.plan()
    assert abs(plan.root_x0 + 0.5) < 1e-9 and abs(plan.root_y0 + 0.5) < 1e-9
    a = w.nodes
    c = 0.5 * (a + np.roll(a, -1, axis=0))
    h = float(np.linalg.norm(a[1] - a[0]))
    cs, sn = math.cos(w.theta), math.sin(w.theta)
    far = (0.0625 * math.sqrt(2.0) + 0.5 * h) * 10 ** 0.7          # where the cut at 10^-14.7 began
    dx = math.sqrt(far * far - 0.0625 ** 2)
    worst = 0.0
    for i in range(w.E):
        psi = np.zeros(2 * w.E, np.complex128)
        psi[2 * i] = 1e8                                    # the incident field's derivative is lost beside it
        for x1 in math.copysign(0.0625, c[i, 0]) + dx + np.linspace(1e-6, 0.004, 6):
            du = np.zeros(1, np.complex128)
            pf.pfmbem_field_dx1(s.h, psi, np.array([[x1, 0.0]]), None, du)
            inc = 1j * w.k * cs * np.exp(1j * w.k * cs * x1)
            r = math.hypot(x1 - c[i, 0], c[i, 1])
            worst = max(worst, abs(pf.pfmbem_etc(s.h, psi, float(x1), 1) * w.k - abs(du[0] + inc))
                        / (1e8 * h / (2 * math.pi * r * r)))
    s.close()
    assert worst < 1e-14, worst
