"""The triangle tree's cached product is as accurate as its tables: its sums over the near
field, the same fiber, the cells and L2P are FP64 sums, and only the translations between
boxes run in double-float words."""
import math

import pytest
import torch

from paper_1910_10863_gb300 import workloads as W
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu


def handle(pf, cols, rows, n, kH):
    w = W.hexagon_block(cols, rows, 1.0, n, kH, math.radians(23.0), seed=9)
    return w, pf.Solver(w, tree=1, leaf_max=16, **W.hexagon_block_lattice(1.0, rows))


@pytest.mark.parametrize("cols,rows,n,kH", [(3, 3, 43, 1.0), (4, 5, 176, 5.1), (2, 4, 222, 7.6), (5, 8, 61, 3.5)])
def test_rounding_of_the_product(cols, rows, n, kH):
    """x and x times 1 + 2^-26 (which an FP32 pair holds to other bits): the products' ratio is that of the vectors up
    to both products' rounding.  FP64 sums of up to 5000 terms round to sqrt(5000) 2^-53 of their size, the far field's
    double-float sums (48 bits, up to a tenth of the result) to 1e-15: 4e-15 of the result."""
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    w, s = handle(pf, cols, rows, n, kH)
    g = torch.Generator(device="cuda").manual_seed(4)
    f = 1.0 + 2.0 ** -26
    worst = []
    for _ in range(4):
        x = torch.randn(2 * s.E, dtype=torch.complex128, device="cuda", generator=g)
        # 26 bits less in x, so that x f is exact
        x = torch.complex(x.real.float().double(), x.imag.float().double())
        y, z = torch.zeros_like(x), torch.zeros_like(x)
        s.matvec(x, y, pf.FP64)
        s.matvec(x * f, z, pf.FP64)
        torch.cuda.synchronize()
        worst.append(float((z - f * y).norm() / y.norm()))
    s.close()
    assert max(worst) < 4e-15, worst
