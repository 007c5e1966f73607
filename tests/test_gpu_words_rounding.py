"""The square tree's FP64 product in double-float words is no further from the same product in
FP64 arithmetic (one kernel per stage) than it was with L2P, the multipoles between the stages
and the phases in FP64."""
import numpy as np
import pytest
import torch

from paper_1910_10863_gb300 import workloads as W
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu

# block and the relative difference that it had then (median over these 40 vectors)
CASES = [("square", 2, 2, 64, 2.0, 4.38e-15), ("square", 3, 5, 33, 4.0, 3.90e-15), ("square", 2, 2, 17, 0.7, 3.22e-15),
         ("square", 1, 1, 33, 1.0, 2.58e-15), ("square", 1, 2, 200, 1.0, 6.82e-15),
         ("square", 16, 16, 64, 10.0, 1.015e-14), ("hexagon", 2, 3, 33, 1.0, 4.82e-15),
         ("hexagon", 4, 4, 97, 5.0, 3.68e-15), ("hexagon", 8, 8, 256, 5.0, 4.50e-15)]


@pytest.mark.parametrize("lattice,cols,rows,n,kH,limit", CASES)
def test_rounding_is_no_larger(lattice, cols, rows, n, kH, limit):
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    w = W.hexagon_block(cols, rows, 1.0, n, kH, 0.4, 9) if lattice == "hexagon" else \
        W.square_block(cols, rows, 1.0, 0.25, n, kH, 0.4)
    s, r = pf.Solver(w), pf.Solver(w, launch=1)
    g = torch.Generator(device="cuda").manual_seed(4)
    d = []
    for _ in range(40):
        x = torch.randn(2 * s.E, dtype=torch.complex128, device="cuda", generator=g)
        y, z = torch.zeros_like(x), torch.zeros_like(x)
        s.matvec(x, y, pf.FP64)
        r.matvec(x, z, pf.FP64)
        torch.cuda.synchronize()
        d.append(float((y - z).norm() / z.norm()))
    s.close()
    r.close()
    assert np.median(d) < limit, (np.median(d), limit)
