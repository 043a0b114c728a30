"""GPU: the one-launch 2D step (FD of a step and collide of the next in one
kernel) against the oracle and against itself cut differently.

Bounds: FP32 deviations |d phi| <= 1e-5 and |d u*| <= 1e-3 max|u*| (the stated
FP32 bar, here after a few steps).  Cuts of one run agree bitwise: every
operation of the kernel is explicitly rounded."""
import numpy as np
import pytest

import oracle as O
from paper_0902_3921_gb300 import lbm

pytestmark = pytest.mark.gpu

CFG = dict(a=-0.1, b=0.1, kappa=0.14, tau=0.9, Gamma=0.5, N=0.3, Q=2.5)


def _fields(Lx, Ly):
    rng = np.random.default_rng(Lx * 1000 + Ly)
    x, y = np.arange(Lx) / Lx, np.arange(Ly)[:, None] / Ly
    phi = 0.6 * np.cos(2 * np.pi * (x + y)) + 0.2 * (rng.random((Ly, Lx)) - 0.5)
    n = 1 + 0.01 * (rng.random((Ly, Lx)) - 0.5)
    u = np.stack([0.03 * np.sin(2 * np.pi * y) + 0 * x, 0.03 * np.cos(2 * np.pi * x) + 0 * y])
    return n, phi, u


# lattices under a tile and its halo (the region wraps several times), whole
# tiles, one site over, Lx no multiple of 4
@pytest.mark.parametrize("Lx,Ly", [(3, 4), (32, 16), (64, 64), (33, 17), (100, 37), (129, 66)])
@pytest.mark.parametrize("rows", [16, 32])
@pytest.mark.parametrize("form", ["m4", "flux", "m1", "m2_half_force", "m3_flux"])
def test_against_oracle(Lx, Ly, rows, form, monkeypatch):
    monkeypatch.setenv("HLBM_TUNING", f"4,{rows},4,2,2")
    kw, m = dict(CFG), 4
    if form in ("flux", "m3_flux"):
        kw["adv_variant"] = 1
    if form.startswith("m"):
        m = int(form[1])
    if form in ("m1", "m2_half_force", "m3_flux"):
        kw["Gamma"] = 0.05  # stable at small m
    if form == "m2_half_force":
        kw.update(cubic_at_half=1, g=(1e-4, -2e-4, 0.0), force_steps=3)
    n, phi, u = _fields(Lx, Ly)
    ref = O.State.create(O.Params(Lx=Lx, Ly=Ly, m=m, **kw), n, phi, u)
    ref.run(6)
    lat = lbm.Lattice(lbm.LbmParams(Lx=Lx, Ly=Ly, fd_substeps=-m, precision=lbm.LBM_F32DEV, **kw)).init_fields(n, phi, u)
    lat.step(6)
    assert lbm.lbm_tuning(lat.handle)["fd_tile_width"] == 2
    gn, gphi, gu = lat.moments()
    rn, ru = ref.moments()
    umax = np.max(np.sqrt(np.sum(ru * ru, axis=0)))
    assert np.max(np.abs(gphi - ref.phi)) <= 1e-5
    assert np.max(np.abs(gu - ru)) <= 1e-3 * umax
    lat.close()


@pytest.mark.parametrize("rows", [16, 32])
def test_cuts_of_a_run_agree_bitwise(rows, monkeypatch):
    """One lbm_step call (with a force that ends inside it), single steps,
    plain launches and launches timed one by one: the same populations, phi
    and u* planes."""
    import torch
    monkeypatch.setenv("HLBM_TUNING", f"4,{rows},4,5,2")
    Lx, Ly = 136, 70
    p = lbm.LbmParams(Lx=Lx, Ly=Ly, precision=lbm.LBM_F32DEV, g=(1e-4, 0.0, 0.0), force_steps=4, **CFG)
    out = []
    for cuts, graphs, timing in (([9], True, False), ([1] * 9, True, False), ([2, 7], False, False),
                                 ([9], True, True)):
        bufs = {"populations": [torch.zeros(9, Ly, Lx, device="cuda") for _ in range(2)],
                "phi": [torch.zeros(Ly, Lx, device="cuda") for _ in range(3)],
                "u": torch.zeros(2, Ly, Lx, device="cuda")}
        lat = lbm.Lattice(p, buffers=bufs)
        lbm.lbm_set_graphs(lat.handle, graphs)
        lbm.lbm_set_kernel_timing(lat.handle, timing)
        lat.init_fields(*_fields(Lx, Ly))
        for c in cuts:
            lat.step(c)
        lat.synchronize()
        out.append((bufs["populations"][1].clone(), bufs["phi"][1].clone(), bufs["u"].clone()))
        lat.close()
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert torch.equal(a, b)
