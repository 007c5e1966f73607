"""Triangle-tree handles of different sizes, each used by its own host thread: a kernel's
limit of dynamic shared memory belongs to the process, and no handle's product may lower it
between another's setting and its launch."""
import math
import threading

import pytest
import torch

from paper_1910_10863_gb300 import workloads as W
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu


def test_products_of_two_sizes_at_the_same_time():
    """Fibers of 1000 and of 520 elements (96 and 50 KB of the same-fiber kernel) at orders 30 and 24 of the
    M2L: 1500 products a thread, all with status 0, the last equal to the first."""
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    lat = W.hexagon_block_lattice(1.0, 2)
    made, errors = [], []
    for n, p in ((1000, 30), (520, 24)):
        w = W.hexagon_block(2, 2, 1.0, n, 2.0, math.radians(20.0), seed=3)
        s = pf.Solver(w, tree=1, leaf_max=64, p=p, **lat)
        assert s.plan().near_blocks > 0
        g = torch.Generator(device="cuda").manual_seed(n)
        x = torch.randn(2 * s.E, dtype=torch.complex128, device="cuda", generator=g)
        y = torch.zeros_like(x)
        s.matvec(x, y, pf.FP64)
        made.append((s, x, y))
    torch.cuda.synchronize()
    first = [y.clone() for _, _, y in made]

    def work(s, x, y):
        try:
            for _ in range(1500):
                s.matvec(x, y, pf.FP64)
        except Exception as e:
            errors.append(e)

    ts = [threading.Thread(target=work, args=m) for m in made]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for (s, _, y), f in zip(made, first):
        assert float((y - f).norm() / f.norm()) < 1e-12
        s.close()
