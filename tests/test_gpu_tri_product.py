"""The triangle tree's cached product (double-float words, two streams) against the same
tree with the element integrals in every product and FP64 translations: fibers with and
without a circulant block, odd element counts, one to several levels, leaves of one and
of many elements, expansion orders at both sides of a warp, and one stream (profile)."""
import math

import numpy as np
import pytest
import torch

from paper_1910_10863_gb300 import workloads as W
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu

CASES = [
    ("poly", 3, 3, 33, 3.0, {"leaf_max": 16}),
    ("poly", 3, 3, 33, 3.0, {"depth": 4}),
    ("poly", 4, 4, 97, 5.0, {"leaf_max": 40}),
    ("poly", 4, 4, 97, 5.0, {"depth": 5}),
    ("poly", 3, 4, 255, 2.0, {"leaf_max": 16}),
    ("poly", 2, 3, 64, 2.0, {"p": 15}),
    ("poly", 2, 3, 64, 2.0, {"p": 16}),
    ("poly", 2, 3, 64, 2.0, {"p": 52}),
    ("poly", 2, 3, 64, 2.0, {"leaf_max": 16, "profile": 1}),
    ("roundsquare", 4, 6, 64, 0.62, {"leaf_max": 16}),
]


@pytest.mark.parametrize("kind,cols,rows,n,f,opts", CASES)
def test_cached_product_matches_integrals(kind, cols, rows, n, f, opts):
    """Tolerance: sums of up to some thousand terms of 48 bits with up to three digits of
    cancellation, and the Gauss ladder's 1e-14 an element: 1e-11 of the result."""
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    if kind == "poly":
        w = W.hexagon_block(cols, rows, 1.0, n, f, math.radians(23.0), seed=9)
        lat = W.hexagon_block_lattice(1.0, rows)
    else:
        w = W.table3_block(f, f=0.35, lattice="hexagon", scatterer=kind, n=n)
        lat = W.table3_hexagon_lattice()
    base = dict(opts)
    base.pop("profile", None)
    s = pf.Solver(w, tree=1, **lat, **opts)
    r = pf.Solver(w, tree=1, near_mode=1, **lat, **base)
    assert s.plan().near_blocks > 0 and r.plan().near_blocks == 0
    g = torch.Generator(device="cuda").manual_seed(4)
    xs = [torch.randn(2 * s.E, dtype=torch.complex128, device="cuda", generator=g) for _ in range(3)]
    ys = [torch.full_like(x, 7.0) for x in xs]
    for _ in range(2):                     # back to back: each product waits for the one before on both streams
        for x, y in zip(xs, ys):
            s.matvec(x, y, pf.FP64)
    for x, y in zip(xs, ys):
        ref = torch.zeros_like(x)
        r.matvec(x, ref, pf.FP64)
        torch.cuda.synchronize()
        assert float((y - ref).norm() / ref.norm()) < 1e-11
    s.close()
    r.close()
