"""Batched solves of fewer instances than groups of the default size: the chip in equal
shares (one instance on all of it, a share that does not divide it, shares at both sides
of the default), and the default where instances are many; each against its own solve."""
import numpy as np
import pytest

from paper_1910_10863_gb300 import workloads as W
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,group", [(1, 0), (2, 0), (7, 0), (33, 0), (39, 0), (2, 8)])
def test_shares_match_single_solves(count, group):
    """Tolerance: both residuals below 1e-6 and condition numbers of up to some hundred: 5e-4 of the solution."""
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    ss = [pf.Solver(w, precision=pf.MIXED, batch_group=group) for w in W.batch_instances(count, seed=7)]
    psis = [np.zeros(2 * s.E, np.complex128) for s in ss]
    st, infos = pf.pfmbem_solve_batch([s.h for s in ss], psis, tol=1e-6)
    assert st == 0 and all(i.status == 0 and i.rel_residual <= 1e-6 for i in infos)
    for s, p in zip(ss, psis):
        ref = np.zeros_like(p)
        s.solve(ref, tol=1e-6)
        assert np.linalg.norm(p - ref) < 5e-4 * np.linalg.norm(ref)
        s.close()
