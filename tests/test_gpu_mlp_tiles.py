"""The network's products at the edges of their tiles (32 x 32 with K stages of 128, and
64 x 64 with K stages of 32): one row to more than a tile of rows, widths below, at and
above a tile, batches that take the large tile forward and backward; host and device
buffers, and a device batch at an odd offset.  Against the FP64 oracle."""
import numpy as np
import pytest

from oracle import mlp as omlp
from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu

CASES = [  # inputs, hidden, layers, outputs, batch
    (1, 1, 1, 1, 1), (3, 5, 2, 7, 2), (50, 256, 3, 1088, 15), (50, 256, 3, 68, 129), (33, 64, 1, 31, 257),
    (17, 127, 2, 129, 16), (50, 256, 3, 1088, 1090), (50, 256, 2, 33, 4097), (64, 512, 1, 64, 2049)]


def params(rng, dims):
    out = []
    for i, o in zip(dims[:-1], dims[1:]):
        out += [rng.uniform(-1, 1, i * o) * np.sqrt(3.0 / i), 0.1 * rng.standard_normal(o)]
    return np.concatenate(out).astype(np.float32)


@pytest.mark.parametrize("n_in,hidden,layers,n_out,batch", CASES)
def test_tiles_match_oracle(n_in, hidden, layers, n_out, batch):
    """Tolerance: FP32 sums of at most 4097 products of order one, eps_32 sqrt(K) = 4e-6 of the largest entry
    through up to four layers: 2e-5 of the norm."""
    import torch
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem as pf
    rng = np.random.default_rng(batch + n_out)
    dims = [n_in] + [hidden] * layers + [n_out]
    p = params(rng, dims)
    X = rng.standard_normal((batch, n_in)).astype(np.float32)
    T = rng.standard_normal((batch, n_out)).astype(np.float32)
    lo, go = omlp.loss_and_grad(p.astype(np.float64), dims, X.astype(np.float64), T.astype(np.float64))
    a, o = X.astype(np.float64), 0
    from math import sqrt

    from scipy.special import erf
    for l, (i, n) in enumerate(zip(dims[:-1], dims[1:])):
        a = a @ p[o:o + i * n].reshape(n, i).T.astype(np.float64) + p[o + i * n:o + i * n + n]
        o += i * n + n
        if l < layers:
            a = 0.5 * a * (1 + erf(a / sqrt(2)))
    net = pf.MLP(n_in, hidden, layers, n_out)
    net.set_params(p)
    loss, g = net.train(X, T, lr=0.0, want_grad=True)
    Y = net.forward(X)
    # device buffers, the batch at an offset of one float
    Xd = torch.empty(batch * n_in + 1, device="cuda")[1:].view(batch, n_in)
    Xd.copy_(torch.from_numpy(X))
    Td, gd = torch.from_numpy(T).cuda(), torch.zeros(len(p), device="cuda")
    Yd = net.forward(Xd, torch.zeros(batch, n_out, device="cuda"))
    st = pf.lib().pfmbem_mlp_train(net.h, batch, pf.addr(Xd), pf.addr(Td), 0.0, None, pf.addr(gd))
    assert st == 0
    torch.cuda.synchronize()
    assert abs(loss - lo) < 2e-5 * abs(lo)
    for v in (g, gd.cpu().numpy()):
        assert np.linalg.norm(v - go) < 2e-5 * np.linalg.norm(go)
    for v in (Y, Yd.cpu().numpy()):
        assert np.linalg.norm(v - a) < 2e-5 * np.linalg.norm(a)
