"""GPU: the autotuner's choice is kept per scheme: a stencil_fd handle created
after a printed-form handle of the same shape and m must not take its FD
kernel (only the tile kernel evaluates the stencil operators)."""
import numpy as np
import pytest

import oracle as O
from paper_0902_3921_gb300 import inputs as I
from paper_0902_3921_gb300 import lbm

pytestmark = pytest.mark.gpu


def test_stencil_handle_after_a_printed_one():
    kw = dict(a=-0.1, b=0.1, kappa=0.14, tau=1.0, Gamma=0.5, N=0.3, Q=2.5)
    Lx, Ly, m = 140, 76, 21
    lp = dict(Lx=Lx, Ly=Ly, fd_substeps=m, precision=lbm.LBM_F32DEV, **kw)
    lbm.Lattice(lbm.LbmParams(**lp)).close()
    op = O.Params(Lx=Lx, Ly=Ly, m=m, stencil_fd=1, **kw)
    phi = I.drop(2, Lx, Ly, R=15, phi0=O.phi0_of(op), xi=O.xi_of(op))
    n, u = I.rest(2, Lx, Ly)
    ref = O.State.create(op, n, phi, u)
    ref.run(10)
    lat = lbm.Lattice(lbm.LbmParams(stencil_fd=1, **lp)).init_fields(n, phi, u).step(10)
    assert lbm.lbm_tuning(lat.handle)["fd_tile_width"] in (32, 64)
    assert np.max(np.abs(lat.moments()[1] - ref.phi)) <= 1e-5
    lat.close()
