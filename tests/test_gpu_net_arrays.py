"""GPU: the surrogate's state arrays at any float alignment and in any overlap.

A view that starts one float into a buffer is not 16-byte aligned: prediction,
loss and gradients must be those of the aligned arrays, bitwise (the arithmetic
does not depend on how the floats are loaded).  A prediction into an array that
overlaps its input (frames t .. t + N - 1 into t + 1 .. t + N, or in place) must be
that of separate arrays."""
import numpy as np
import pytest
import torch

from paper_0902_3921_gb300 import lbm

pytestmark = pytest.mark.gpu

# tcgen05 (1024 tiles and more), mma.sync
SHAPES = [(1, 1024, 128), (2, 264, 256), (2, 64, 64)]


def _net():
    net = lbm.Net(32, 3, seed=3)
    net.set_normalisation([0.01, 0.0, -0.01, 0.0], [0.9, 1.1, 1.0, 1.2], [0.5, 0.25, 0.125, 1.0])
    return net


def _rand(seed, *shape):
    return torch.randn(*shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))


def _offset(t, k):
    buf = torch.zeros(t.numel() + 8, device="cuda")
    v = buf[k:k + t.numel()].view(t.shape)
    v.copy_(t)
    assert v.data_ptr() % 16 == 4 * k % 16
    return v


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("k0,k1", [(1, 0), (0, 1), (3, 2)])
def test_unaligned_views(shape, k0, k1):
    net, (N, H, W) = _net(), shape
    x0 = _rand(H, N, H, W, 4)
    x1 = x0 + 0.5 * _rand(W, N, H, W, 4)
    res = []
    for a, b in ((x0, x1), (_offset(x0, k0), _offset(x1, k1))):
        out = torch.zeros_like(x0) if b is x1 else _offset(torch.zeros_like(x0), k1)
        net.forward(a.data_ptr(), N, H, W, out.data_ptr())
        torch.cuda.synchronize()
        loss = net.train_step(a.data_ptr(), b.data_ptr(), N, H, W, lr=0.0, update=False)
        assert torch.equal(a, x0) and torch.equal(b, x1)
        res.append((out.clone(), loss, net.get_grads().copy()))
    assert torch.equal(res[0][0], res[1][0])
    assert res[0][1] == res[1][1]
    assert np.array_equal(res[0][2], res[1][2])
    net.close()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("shift", ["in place", "frame", "pixel", "float"])
def test_overlapping_output(shape, shift):
    net, (N, H, W) = _net(), shape
    x0 = _rand(H, N, H, W, 4)
    ref = torch.zeros_like(x0)
    net.forward(x0.data_ptr(), N, H, W, ref.data_ptr())
    n, d = x0.numel(), {"in place": 0, "frame": H * W * 4, "pixel": 4, "float": 1}[shift]
    for back in (False, True):  # x1 after or before x0
        buf = torch.zeros(n + d, device="cuda")
        a, b = (buf[d:], buf[:n]) if back else (buf[:n], buf[d:])
        a[:n].copy_(x0.flatten())
        net.forward(a.data_ptr(), N, H, W, b.data_ptr())
        torch.cuda.synchronize()
        assert torch.equal(b[:n].view(x0.shape), ref)
    net.close()
