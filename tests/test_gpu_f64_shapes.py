"""GPU: the FP64 kernels at the lattice shapes where their launch shapes can go
wrong, against the oracle at the FP64 bounds (|d phi|, |d f| <= 1e-11, |d u*| <=
1e-12: FMA contraction and summation order are the only differences)."""
import numpy as np
import pytest

import oracle as O
from paper_0902_3921_gb300 import lbm

pytestmark = pytest.mark.gpu

CFG = dict(a=-0.1, b=0.1, kappa=0.14, tau=0.9, Gamma=0.5)


def _check(dims, shape, steps, m, **kw):
    """Random fields (every neighbour differs) for `steps` LB steps."""
    Lx, Ly, Lz = shape
    kw = dict(CFG, **kw)
    op = O.Params(dims=dims, Lx=Lx, Ly=Ly, Lz=Lz, m=m, **kw)
    lp = lbm.LbmParams(dims=dims, Lx=Lx, Ly=Ly, Lz=Lz, fd_substeps=-m, precision=lbm.LBM_F64, **kw)
    grid = (Lz, Ly, Lx) if dims == 3 else (Ly, Lx)
    rng = np.random.default_rng(Lx * 1000 + Ly)
    phi = 0.8 * (rng.random(grid) - 0.5)
    n = 1 + 0.01 * (rng.random(grid) - 0.5)
    u = 0.02 * (rng.random((dims,) + grid) - 0.5)
    ref = O.State.create(op, n, phi, u)
    ref.run(steps)
    lat = lbm.Lattice(lp).init_fields(n, phi, u).step(steps)
    rn, ru = ref.moments()
    gn, gphi, gu = lat.moments()
    assert np.max(np.abs(gphi - ref.phi)) <= 1e-11
    assert np.max(np.abs(gu - ru)) <= 1e-12
    assert np.max(np.abs(gn - rn)) <= 1e-11
    assert np.max(np.abs(lat.populations() - ref.f)) <= 1e-11
    lat.close()


# sites: under one block of 128, exactly two blocks, ragged; the smallest sides
@pytest.mark.parametrize("shape", [(3, 3, 3), (5, 4, 3), (8, 8, 4), (37, 13, 11)])
@pytest.mark.parametrize("form", ["paper", "flux", "half_T"])
def test_3d(shape, form):
    kw = dict(N=1 / 6, Q=1 / 3)
    if form == "flux":
        kw["adv_variant"] = 1
    elif form == "half_T":
        kw.update(cubic_at_half=1, T=0.3, g=(1e-5, -2e-5, 3e-5), force_steps=2)
    _check(3, shape, 4, 8, **kw)


# the 16 x 8 collide tile with both FD tiles (16 x 8 and 32 x 16): lattices
# smaller than a tile and its halo, whole tiles, one site over
@pytest.mark.parametrize("shape", [(3, 3, 1), (16, 8, 1), (33, 17, 1), (32, 48, 1), (71, 45, 1)])
@pytest.mark.parametrize("rows", [8, 16])
@pytest.mark.parametrize("form", ["paper", "flux", "half_T", "stencil"])
def test_2d(shape, rows, form, monkeypatch):
    monkeypatch.setenv("HLBM_TUNING", f"1,{rows},2,8,32")
    kw, m = dict(N=0.3, Q=2.5), 4
    if form == "flux":
        kw["adv_variant"] = 1
    elif form == "half_T":
        kw.update(cubic_at_half=1, T=0.3, g=(1e-5, -2e-5, 0.0), force_steps=2)
    elif form == "stencil":
        kw["stencil_fd"], m = 1, 21
    _check(2, shape, 4, m, **kw)
