"""GPU: 3D results keep their bits.

FP16 storage rounds a population to the other neighbour where FP32 arithmetic in
another order differs in a last bit, which after a few steps is 1e-4 of the
result, so the 3D kernels keep the operations of a row length and their order:
(a) the step with the fused psi / new-phi kernel equals the step in separate
passes bitwise (rows of 128 and 256 sites excepted, whose order is their own);
(b) phi and the populations of short FP16 runs equal recorded digests."""
import hashlib

import numpy as np
import pytest

from paper_0902_3921_gb300 import lbm

pytestmark = pytest.mark.gpu

CFG = dict(a=-0.1, b=0.1, kappa=0.14, tau=0.9, Gamma=0.5, N=1 / 6, Q=1 / 3)


def _run(shape, precision, flux, steps=3, m=8, **kw):
    """Random fields from IEEE additions and products only (the same bits on any host)."""
    Lx, Ly, Lz = shape
    rng = np.random.default_rng(Lx * 100 + Ly)
    grid = (Lz, Ly, Lx)
    n = 1 + 0.01 * (rng.random(grid) - 0.5)
    phi = 0.8 * (rng.random(grid) - 0.5)
    u = 0.05 * (rng.random((3,) + grid) - 0.5)
    lat = lbm.Lattice(lbm.LbmParams(dims=3, Lx=Lx, Ly=Ly, Lz=Lz, fd_substeps=-m, precision=precision,
                                    adv_variant=flux, cubic_at_half=flux, **dict(CFG, **kw)))
    lat.init_fields(n, phi, u).step(steps)
    out = lat.moments()[1].copy(), lat.populations().copy()
    lat.close()
    return out


# one quad to 64 a row, an odd quad count, several rows to a warp
@pytest.mark.parametrize("shape", [(4, 5, 3), (12, 7, 9), (36, 33, 6), (68, 40, 5), (100, 17, 9), (132, 16, 8),
                                   (200, 15, 10)])
@pytest.mark.parametrize("flux", [0, 1])
@pytest.mark.parametrize("precision", [lbm.LBM_F32DEV, lbm.LBM_F16DEV])
def test_fused_kernel_equals_passes(shape, flux, precision, monkeypatch):
    fused = _run(shape, precision, flux)
    monkeypatch.setenv("HLBM_FD3_UNFUSED", "1")
    for a, b in zip(fused, _run(shape, precision, flux)):
        assert np.array_equal(a, b)


DIGESTS = {
    ((12, 7, 9), "paper"): "bc48fc767541626405122d7a4bed1590",
    ((12, 7, 9), "flux"): "44c0d31b8b1ac960b7ead6453ef09abb",
    ((12, 7, 9), "T"): "d72a1b91ef1f3858c6e39f5d1bd30403",
    ((12, 7, 9), "m3"): "890b34a336fa9960b967f507038ceb58",
    ((37, 13, 11), "paper"): "e5d11e2d803111e0304989577218c6d3",
    ((37, 13, 11), "flux"): "c8202b958897265dfb462d9d2b2999e1",
    ((37, 13, 11), "T"): "e352bf71e2486be9eb6686c15b6d80a7",
    ((37, 13, 11), "m3"): "dff7e4cf0de7346961410b930c1097a1",
    ((100, 17, 9), "paper"): "9b64a7e183bb7729df95bb6a7c9cf940",
    ((100, 17, 9), "flux"): "f25d56ab870353e5c0326e02b608a3f9",
    ((100, 17, 9), "T"): "3c99180b20990cddb9dcf82f46bf32b3",
    ((100, 17, 9), "m3"): "0628b5390e8bba98421dc4675aa6111d",
    ((128, 10, 9), "paper"): "93fd0f269f20ddb0c214800e1bebbc53",
    ((128, 10, 9), "flux"): "1878533556445da697f85cc772ef27ec",
    ((128, 10, 9), "T"): "8f888f463d2369abe04e6ae4081f35a2",
    ((128, 10, 9), "m3"): "b49f7cb62bff6fb6fd261ed636afa87a",
    ((196, 9, 10), "paper"): "6d274f30a16e0219e5a094183f7e3d83",
    ((196, 9, 10), "flux"): "cc3224822daec526264b5aeaa185c84b",
    ((196, 9, 10), "T"): "24b1098adb8a5b7c25ec76c7bf743ddb",
    ((196, 9, 10), "m3"): "01d68704f7e7ad81e0168384df819e4f",
    ((256, 9, 8), "paper"): "2e07f8b83562747fa68957b77f21dcba",
    ((256, 9, 8), "flux"): "116ab795345881ec2633e5c2d916632f",
    ((256, 9, 8), "T"): "6c871e8c62a1f600486fdd0c3b43d768",
    ((256, 9, 8), "m3"): "daad70fd72eb43fa81d879e189c70751",
    ((260, 6, 9), "paper"): "5ae7718b2843af7e868a8e6b434ad65f",
    ((260, 6, 9), "flux"): "a667933b674f878936047ad5e88c6345",
    ((260, 6, 9), "T"): "4b6a794a05140610d39c8ca1337ca119",
    ((260, 6, 9), "m3"): "6f1af4d3978390cd0b1ecbfbbc8f2a33",
}


def digest(shape, form):
    kw = {"T": dict(T=0.3, g=(1e-5, -2e-5, 3e-5), force_steps=2), "m3": dict(m=3, Gamma=0.15)}.get(form, {})
    out = _run(shape, lbm.LBM_F16DEV, 1 if form == "flux" else 0, **kw)
    return hashlib.sha256(b"".join(np.ascontiguousarray(a).tobytes() for a in out)).hexdigest()[:32]


FORMS = ("paper", "flux", "T", "m3")
SHAPES = ((12, 7, 9), (37, 13, 11), (100, 17, 9), (128, 10, 9), (196, 9, 10), (256, 9, 8), (260, 6, 9))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("form", FORMS)
def test_f16_digest(shape, form):
    assert digest(shape, form) == DIGESTS[shape, form]
