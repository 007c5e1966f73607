"""The triangle tree's cached product at orders whose M2L operators exceed the shared memory that the grouped
form takes (53 and up): such a level goes target by target, with L2L, after the grouped form of the others."""
import math

import pytest
import torch

from paper_1910_10863_gb300 import workloads as W
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [{"p": 53}, {"p": 60}, {"p": 54, "depth": 3}])
def test_levels_by_lists(opts):
    """Against the same tree with the element integrals in every product and FP64 translations: sums of 48 bits
    with up to three digits of cancellation and the Gauss ladder's 1e-14 an element, 1e-11 of the result."""
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    w = W.hexagon_block(2, 3, 1.0, 64, 2.0, math.radians(23.0), seed=9)
    lat = W.hexagon_block_lattice(1.0, 3)
    s = pf.Solver(w, tree=1, **lat, **opts)
    r = pf.Solver(w, tree=1, near_mode=1, **lat, **opts)
    assert s.plan().near_blocks > 0 and r.plan().near_blocks == 0
    g = torch.Generator(device="cuda").manual_seed(4)
    for _ in range(3):
        x = torch.randn(2 * s.E, dtype=torch.complex128, device="cuda", generator=g)
        y, z = torch.full_like(x, 7.0), torch.zeros_like(x)
        s.matvec(x, y, pf.FP64)
        r.matvec(x, z, pf.FP64)
        torch.cuda.synchronize()
        assert float((y - z).norm() / z.norm()) < 1e-11
    s.close()
    r.close()
