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


def test_step_with_a_device_gradient(pf):
    """Adam reads the gradient where the pass wrote it, in the caller's buffer or the network's own: the same parameters
    bit for bit after three steps."""
    import torch
    X, T = batch(1)
    out = []
    for where in ("device", "host", "none"):
        net = pf.MLP(N_IN, HIDDEN, LAYERS, N_OUT, seed=5)
        p = net.get_params()
        g = {"device": torch.zeros(len(p), device="cuda"), "host": np.zeros(len(p), np.float32), "none": None}[where]
        for _ in range(3):
            assert train(pf, net, X, T, lr=1e-3, grad=g) == 0
        q = net.get_params()
        assert np.abs(q - p).max() > 1e-4
        out.append(q)
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])


def test_buffers_that_share_memory(pf):
    """An output over the input, and a gradient over the batch: as with buffers of their own."""
    import torch
    net = pf.MLP(N_IN, HIDDEN, LAYERS, N_OUT)
    X, T = batch(2)
    n = net.nparams()
    Y, G = torch.zeros(BATCH, N_OUT, device="cuda"), torch.zeros(n, device="cuda")
    assert pf.lib().pfmbem_mlp_forward(net.h, BATCH, pf.addr(X), pf.addr(Y)) == 0
    assert train(pf, net, X, T, grad=G) == 0
    for at in (0, 5, BATCH * N_IN - 1):                    # Y from X's first, fifth, last entry on
        buf = torch.zeros(BATCH * (N_IN + N_OUT), device="cuda")
        buf[:X.numel()] = X.flatten()
        torch.cuda.synchronize()
        assert pf.lib().pfmbem_mlp_forward(net.h, BATCH, buf.data_ptr(), buf.data_ptr() + 4 * at) == 0
        torch.cuda.synchronize()
        assert torch.equal(buf[at:at + Y.numel()].view_as(Y), Y)
    for first in (X, T):                                   # the gradient over X, then over T
        buf = torch.zeros(max(n, first.numel()), device="cuda")
        buf[:first.numel()] = first.flatten()
        a = (buf, T) if first is X else (X, buf)
        assert train(pf, net, a[0], a[1], grad=buf) == 0
        assert torch.equal(buf[:n], G)
