"""GPU: the 3D FP32 FD path at row lengths where its lane maps can go wrong
(rows of one quad to 64, several rows to a warp, an odd quad count with two
quads a lane, rows past 256 on the three-pass path), one LB step of m = 8
substeps against the oracle at the FP32 bar (|d phi| <= 1e-5, |d u*| <= 1e-3
max|u*|)."""
import numpy as np
import pytest

import oracle as O
from paper_0902_3921_gb300 import lbm

pytestmark = pytest.mark.gpu

CFG = dict(a=-0.1, b=0.1, kappa=0.14, tau=1.0, Gamma=0.5, N=1 / 6, Q=1 / 3)


@pytest.mark.parametrize("shape", [(4, 5, 3), (12, 7, 9), (32, 70, 5), (36, 33, 6), (64, 31, 7), (68, 40, 5),
                                   (100, 17, 9), (132, 16, 8), (196, 9, 7), (200, 15, 10), (260, 6, 5)])
@pytest.mark.parametrize("flux", [0, 1])
def test_rows(shape, flux):
    Lx, Ly, Lz = shape
    grid = (Lz, Ly, Lx)
    rng = np.random.default_rng(Lx)
    phi = 0.8 * (rng.random(grid) - 0.5)
    n = 1 + 0.01 * (rng.random(grid) - 0.5)
    u = 0.05 * (rng.random((3,) + grid) - 0.5)
    kw = dict(CFG, adv_variant=flux, cubic_at_half=flux)
    ref = O.State.create(O.Params(dims=3, Lx=Lx, Ly=Ly, Lz=Lz, m=8, **kw), n, phi, u)
    ref.run(2)
    lat = lbm.Lattice(lbm.LbmParams(dims=3, Lx=Lx, Ly=Ly, Lz=Lz, fd_substeps=-8, precision=lbm.LBM_F32DEV, **kw))
    lat.init_fields(n, phi, u).step(2)
    _, gphi, gu = lat.moments()
    _, ru = ref.moments()
    assert np.max(np.abs(gphi - ref.phi)) <= 1e-5
    assert np.max(np.abs(gu - ru)) <= 1e-3 * np.max(np.sqrt(np.sum(ru * ru, axis=0)))
    lat.close()
