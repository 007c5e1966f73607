"""The buffers that the network's calls accept: a loss in device memory, any alignment, shared memory."""
import numpy as np
import pytest

from tests.gpu_common import ensure_built

pytestmark = pytest.mark.gpu

N_IN, HIDDEN, LAYERS, N_OUT, BATCH = 17, 40, 2, 23, 33


@pytest.fixture(scope="module")
def pf():
    ensure_built()
    from paper_1910_10863_gb300 import pfmbem
    return pfmbem


def batch(seed=0):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    X = torch.randn(BATCH, N_IN, device="cuda", generator=g)
    return X, torch.randn(BATCH, N_OUT, device="cuda", generator=g)


def train(pf, net, X, T, lr=0.0, loss=None, grad=None):
    import torch
    torch.cuda.synchronize()
    st = pf.lib().pfmbem_mlp_train(net.h, BATCH, pf.addr(X), pf.addr(T), lr, pf.addr(loss), pf.addr(grad))
    torch.cuda.synchronize()
    return st


def test_loss_in_device_memory(pf):
    """The loss is copied to the caller's address, which may lie on the device, as a gradient's may.  Its sum's
    order differs from run to run (atomic sums of FP32): 1e-6."""
    import torch
    net = pf.MLP(N_IN, HIDDEN, LAYERS, N_OUT)
    X, T = batch()
    d, h = torch.zeros(1, device="cuda"), np.zeros(1, np.float32)
    assert train(pf, net, X, T, loss=d) == 0
    assert train(pf, net, X, T, loss=h) == 0
    assert h[0] > 0 and abs(d.item() - h[0]) < 1e-6 * h[0]


def test_unaligned_device_buffers(pf):
    """Batches, outputs and gradients at any byte of a device buffer, as copies take them: the same results
    bit for bit as at an aligned address."""
    import torch
    net = pf.MLP(N_IN, HIDDEN, LAYERS, N_OUT)
    X, T = batch(3)
    n = net.nparams()

    def shifted(count, src=None):
        raw = torch.zeros(4 * count + 2, dtype=torch.uint8, device="cuda")
        if src is not None:
            raw[2:].copy_(src.contiguous().view(torch.uint8).flatten())
        return raw, raw.data_ptr() + 2

    def back(raw):
        return raw[2:].clone().view(torch.float32)

    Y, G = torch.zeros(BATCH, N_OUT, device="cuda"), torch.zeros(n, device="cuda")
    assert pf.lib().pfmbem_mlp_forward(net.h, BATCH, pf.addr(X), pf.addr(Y)) == 0
    assert train(pf, net, X, T, grad=G) == 0
    xr, xp = shifted(X.numel(), X)
    tr, tp = shifted(T.numel(), T)
    yr, yp = shifted(Y.numel())
    gr, gp = shifted(n)
    torch.cuda.synchronize()
    assert pf.lib().pfmbem_mlp_forward(net.h, BATCH, xp, yp) == 0
    assert train(pf, net, xp, tp, grad=gp) == 0
    assert torch.equal(back(yr).view_as(Y), Y) and torch.equal(back(gr), G)
