"""ETC, whose derivative goes through the tree's multipoles, against the directly summed
derivative at the same points, over the forms that it accepts: square and triangle
trees, cached and not, blocks wider than their period, deep trees, and the orders and
elements for which ETC is summed directly too."""
import math

import numpy as np
import pytest

from paper_1910_10863_gb300 import workloads as W
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu

HEX = W.hexagon_block(4, 4, 1.0, 20, 3.0, math.radians(17.0), seed=5)
FINE = W.hexagon_block(4, 4, 1.0, 97, 3.0, math.radians(17.0), seed=6)
TRI = W.hexagon_block_lattice(1.0, 4)
CASES = [
    (W.square_block(2, 2, 1.0, 0.3, 64, 2.0, 0.5), {}),
    (W.square_block(2, 2, 1.0, 0.3, 64, 2.0, 0.5), {"depth": 4}),
    (HEX, {"depth": 5}),                              # elements longer than a quarter of a leaf: summed directly
    (FINE, {}),
    (FINE, {"p": 20}),
    (FINE, {"p_min": 12}),                            # orders below 20: summed directly
    (FINE, {"near_mode": 1}),
    (FINE, {"launch": 1}),
    (FINE, dict(tree=1, leaf_max=16, **TRI)),
    (FINE, dict(tree=1, leaf_max=40, near_mode=1, **TRI)),
    (W.square_block(3, 2, 1.0, 0.3, 40, 3.0, math.radians(20)), {}),
    (W.square_block(5, 2, 1.0, 0.3, 64, 2.2, math.radians(35)), {"depth": 4}),
    (W.square_block(4, 4, 1.0, 0.2, 64, 18.0, 0.4), {}),
]


@pytest.mark.parametrize("npts", [1, 300])
@pytest.mark.parametrize("w,opts", CASES, ids=[f"{w.name}-{'-'.join(o) or 'default'}" for w, o in CASES])
def test_etc_matches_direct_derivative(w, opts, npts):
    """Tolerance: a box's expansion ends at 2e-15 of its field, the direct sum's quadrature at 1e-14 of an
    element's, and a random density's terms cancel by up to three digits: 1e-10 of ETC."""
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    s = pf.Solver(w, **opts)
    rng = np.random.default_rng(3)
    psi = rng.standard_normal(2 * w.E) + 1j * rng.standard_normal(2 * w.E)
    plan = s.plan()
    for x1 in (float(np.max(w.centres[:, 0] + w.radii)) + 0.01, float(np.min(w.centres[:, 0] - w.radii)) - 0.05):
        y = plan.root_y0 + w.H * (np.arange(npts) + 0.5) / npts
        pts = np.ascontiguousarray(np.stack([np.full(npts, x1), y], axis=1))
        du = np.zeros(npts, np.complex128)
        pf.pfmbem_field_dx1(s.h, psi, pts, None, du)
        c, sn = math.cos(w.theta), math.sin(w.theta)
        inc = 1j * w.k * c * np.exp(1j * w.k * (c * pts[:, 0] + sn * pts[:, 1]))
        ref = np.mean(np.abs(du + inc)) / w.k
        assert abs(pf.pfmbem_etc(s.h, psi, x1, npts) - ref) < 1e-10 * ref
    s.close()
