"""The element integrals at the edges of the argument ranges of their Bessel
functions (3 and 8): single far elements meet one argument each, so the field of a
small fiber about a point runs through them; against the oracle's own quadrature."""
import math

import numpy as np
import pytest

from oracle import bem
from paper_1910_10863_gb300 import workloads as W
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kH", [0.01, 2.9, 3.1, 7.9, 8.1, 24.5])
def test_field_over_the_argument_ranges(kH):
    """Points at k r from 0.05 kH to 1.2 kH of one fiber (images included).  Tolerance: both sides integrate to
    1e-14 an element and the functions carry 1e-15, the fiber's elements cancel by up to three digits (an
    alternating density): 1e-10 of the largest value; the root's own expansion stays below that within
    0.45 H of the fiber (ratio 0.3 at order 24)."""
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    w = W.single_fiber(0.03, 33, kH, 1.03 * kH, 0.1, 0.3)
    if W.wood_distance(kH, 0.3) < 1e-3:
        pytest.skip("Wood anomaly")
    s = pf.Solver(w)
    rng = np.random.default_rng(1)
    psi = rng.standard_normal(2 * w.E) + 1j * rng.standard_normal(2 * w.E)
    t = np.linspace(0.0, 2 * math.pi, 48, endpoint=False)
    r = np.linspace(0.05, 0.45, 48)
    pts = np.ascontiguousarray(np.stack([r * np.cos(t), r * np.sin(t)], axis=1))
    u = np.zeros(len(pts), np.complex128)
    pf.pfmbem_field(s.h, psi, pts, u)
    ref = bem.potential(bem.problem(w), psi, pts)
    assert np.max(np.abs(u - ref)) < 1e-10 * np.max(np.abs(ref))
