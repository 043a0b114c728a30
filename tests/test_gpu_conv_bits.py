"""GPU: the tcgen05 and the mma.sync convolutions give the same bits, predictions and
(with the same weight-gradient kernel) gradients, so that the choice between them by
image size changes no result: whole and partial 128-pixel tiles, one and several
images, the smallest and deepest nets."""
import numpy as np
import pytest
import torch

from paper_0902_3921_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 8, 128), (2, 48, 256), (1, 512, 256), (1, 8, 144), (2, 40, 160), (3, 24, 368),
                                   (1, 256, 400)])
@pytest.mark.parametrize("C,L", [(32, 2), (32, 6), (16, 3), (16, 8)])
def test_same_bits(shape, C, L, monkeypatch):
    N, H, W = shape
    net = lbm.Net(C, L, seed=5)
    net.set_normalisation([0.0] * 4, [1.0] * 4, [0.5, 0.25, 0.125, 1.0])
    gen = torch.Generator(device="cuda").manual_seed(W)
    x0 = torch.randn(N, H, W, 4, device="cuda", generator=gen)
    x1 = x0 + torch.randn(N, H, W, 4, device="cuda", generator=gen)
    monkeypatch.setenv("HLBM_WGRAD_PATH", "mma")
    out, grads = {}, {}
    for path in ("mma", "tc"):
        monkeypatch.setenv("HLBM_CONV_PATH", path)
        out[path] = torch.zeros_like(x0)
        net.forward(x0.data_ptr(), N, H, W, out[path].data_ptr())
        torch.cuda.synchronize()
        net.train_step(x0.data_ptr(), x1.data_ptr(), N, H, W, lr=0.0, update=False)
        grads[path] = net.get_grads().copy()
    assert not torch.equal(out["tc"], x0)
    assert torch.equal(out["tc"], out["mma"])
    assert np.array_equal(grads["tc"], grads["mma"])
    net.close()
