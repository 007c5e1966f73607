"""The joint Bessel interpolants (ranges to 3, to 8 and beyond) that every element integral of the set-up takes,
through the one call that shows them alone: du/dx1 without u at fewer points than go by leaves is a direct sum of
such integrals.  Against the oracle's analytic derivative of its own quadrature."""
import math

import numpy as np
import pytest

from oracle import bem
from paper_1910_10863_gb300 import workloads as W
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kH", [0.01, 2.9, 3.1, 7.9, 8.1, 24.5])
def test_derivative_over_the_argument_ranges(kH):
    """Points at k r from 0.05 kH to 1.2 kH of one fiber (images included), some of them within 1e-6 of k r = 3 and 8.
    Tolerance: both sides integrate to 1e-13 of an element's derivative, the functions carry 1e-15 and an alternating
    density cancels by up to three digits: 1e-10 of the largest value."""
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    w = W.single_fiber(0.03, 33, kH, 1.03 * kH, 0.1, 0.3)
    assert W.wood_distance(kH, 0.3) > 1e-3
    s = pf.Solver(w)
    rng = np.random.default_rng(1)
    psi = rng.standard_normal(2 * w.E) + 1j * rng.standard_normal(2 * w.E)
    t = np.linspace(0.1, 2 * math.pi, 42, endpoint=False)
    r = np.linspace(0.05, 0.45, 42)
    pts = np.stack([r * np.cos(t), r * np.sin(t)], axis=1)
    # about the element 0's midpoint, at the ranges' edges
    c0 = 0.5 * (w.nodes[0] + w.nodes[1])
    for e in (3.0, 8.0):
        for f in (-1e-6, 0.0, 1e-6):
            if 0.05 < e / kH < 0.45:
                pts = np.concatenate([pts, [[c0[0] + e * (1 + f) / kH, c0[1]]]])
    du = np.zeros(len(pts), np.complex128)
    for a in range(0, len(pts), 24):
        part = np.zeros(min(24, len(pts) - a), np.complex128)
        pf.pfmbem_field_dx1(s.h, psi, np.ascontiguousarray(pts[a:a + 24]), None, part)
        du[a:a + 24] = part
    ref = bem.potential(bem.problem(w), psi, pts, grad=True)[1]
    s.close()
    assert np.max(np.abs(du - ref)) < 1e-10 * np.max(np.abs(ref))
