"""The field's derivative by the leaves' multipoles (32 points and more) against the direct
sums (fewer points in a call) on the same handle: square and triangle trees, blocks wider
than their period, fibers of unequal elements, deep trees, on-the-fly handles, long
wavelengths, densities that radiate and that cancel."""
import math

import numpy as np
import pytest

from paper_1910_10863_gb300 import workloads as W
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu

HEX = W.hexagon_block(4, 4, 1.0, 97, 3.0, math.radians(17.0), seed=6)
CASES = [
    (W.square_block(2, 2, 1.0, 0.3, 64, 2.0, 0.5), {}),
    (W.square_block(2, 2, 1.0, 0.3, 257, 0.01, 0.5), {}),
    (HEX, {}),
    (HEX, {"depth": 5}),
    (HEX, {"near_mode": 1}),
    (HEX, dict(tree=1, leaf_max=16, **W.hexagon_block_lattice(1.0, 4))),
    (W.square_block(5, 2, 1.0, 0.3, 128, 2.2, math.radians(35)), {}),
    (W.square_block(4, 4, 1.0, 0.2, 128, 18.0, 0.4), {}),
    (W.table3_block(0.62, f=0.35, lattice="square", scatterer="roundsquare", n=200), {}),
]


def points(w, count):
    rng = np.random.default_rng(2)
    got = np.empty((0, 2))
    x0, x1 = float(np.min(w.centres[:, 0] - w.radii)) - 0.1 * w.H, float(np.max(w.centres[:, 0] + w.radii)) + 0.1 * w.H
    while len(got) < count:
        p = rng.uniform([x0, -1.5 * w.H], [x1, 2.5 * w.H], size=(4 * count, 2))
        keep = np.ones(len(p), dtype=bool)
        for (cx, cy), r in zip(w.centres, w.radii):
            dy = p[:, 1] - cy
            keep &= np.hypot(p[:, 0] - cx, dy - w.H * np.round(dy / w.H)) > 1.45 * r
        got = np.concatenate([got, p[keep]])
    return np.ascontiguousarray(got[:count])


@pytest.mark.parametrize("smooth", [False, True])
@pytest.mark.parametrize("w,opts", CASES, ids=[f"{i}-{'-'.join(o) or 'default'}" for i, (_, o) in enumerate(CASES)])
def test_leaves_match_direct_sums(w, opts, smooth):
    """Tolerance: a leaf's expansion ends at 1e-15 of its field and rounds some dozen times, the sums of up to 50 k
    terms round too: 1e-13 of the terms' size, which is the elements' sum of |h psi| times the kernels' size at the
    distance of a fifth of a radius (k for H0, its derivative 1/r, the second 1/r^2)."""
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    s = pf.Solver(w, **opts)
    rng = np.random.default_rng(3)
    a = w.nodes
    off = np.concatenate([[0], np.cumsum(w.nodes_per_fiber)])
    nxt = np.arange(len(a)) + 1
    nxt[off[1:] - 1] = off[:-1]
    c, d = 0.5 * (a + a[nxt]), a[nxt] - a
    h = np.hypot(d[:, 0], d[:, 1])
    psi = rng.standard_normal(2 * w.E) + 1j * rng.standard_normal(2 * w.E)
    if smooth:
        dr = np.array([math.cos(w.theta), math.sin(w.theta)])
        psi[0::2] = np.exp(1j * w.k * (c @ dr))
        psi[1::2] = psi[0::2] * ((np.stack([d[:, 1], -d[:, 0]], axis=1) / h[:, None]) @ dr)
    pts = points(w, 75)
    du = np.zeros(75, np.complex128)
    pf.pfmbem_field_dx1(s.h, psi, pts, None, du)
    r = 0.2 * float(np.min(w.radii))
    q = np.sum(h * np.abs(psi[0::2])), np.sum(h * np.abs(psi[1::2])) * w.k
    for i in range(0, 75, 25):
        dv = np.zeros(25, np.complex128)
        pf.pfmbem_field_dx1(s.h, psi, np.ascontiguousarray(pts[i:i + 25]), None, dv)
        assert np.max(np.abs(du[i:i + 25] - dv)) < 1e-13 * (q[0] * (w.k + 1 / r) ** 2 + q[1] * (w.k + 1 / r))
    s.close()
