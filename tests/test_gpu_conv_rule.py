"""GPU: which sizes take the tcgen05 convolution, on both sides of the line: whole
rows, and rows whose partial last tile idles nearly half of the tensor cores'
work.  (The launcher prints its shape under HLBM_CONV_VERBOSE.)"""
import pytest
import torch

from paper_0902_3921_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,shape,tc", [
    (32, (1, 288, 256), False), (32, (1, 304, 256), True), (32, (1, 384, 256), True),
    (32, (1, 512, 144), False), (32, (1, 456, 144), False), (32, (2, 456, 144), True), (32, (1, 360, 272), True),
    (16, (2, 376, 256), False), (16, (2, 472, 256), True), (16, (2, 664, 144), False), (16, (2, 848, 144), False),
    (16, (2, 448, 272), False), (16, (2, 1248, 144), True), (32, (1, 4096, 112), False)])
def test_path_by_size(C, shape, tc, monkeypatch, capfd):
    monkeypatch.setenv("HLBM_CONV_VERBOSE", "1")
    for name in ("HLBM_CONV_PATH", "HLBM_WGRAD_PATH"):
        monkeypatch.delenv(name, raising=False)
    N, H, W = shape
    net = lbm.Net(C, 2, seed=1)
    x0 = torch.zeros(N, H, W, 4, device="cuda")
    net.forward(x0.data_ptr(), N, H, W, x0.data_ptr())
    torch.cuda.synchronize()
    net.close()
    assert (f"{N}x{H}x{W}" in capfd.readouterr().err) == tc
