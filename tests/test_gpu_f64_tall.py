"""GPU: 2D FP64 lattices taller than the 16 x 8 tiles' grid can be (65535 tile rows,
Ly = 524280) are created and stepped, with the tuner's choice and with fixed shapes
that name the small tiles, against the oracle at the FP64 bounds."""
import numpy as np
import pytest

import oracle as O
from paper_0902_3921_gb300 import lbm

pytestmark = pytest.mark.gpu

CFG = dict(a=-0.1, b=0.1, kappa=0.14, tau=0.9, Gamma=0.05, N=0.3, Q=2.5)


def _fields(Lx, Ly):
    rng = np.random.default_rng(Ly)
    return (1 + 0.01 * (rng.random((Ly, Lx)) - 0.5), 0.8 * (rng.random((Ly, Lx)) - 0.5),
            0.02 * (rng.random((2, Ly, Lx)) - 0.5))


@pytest.fixture(scope="module")
def tall():
    Lx, Ly = 3, 524281  # one row over
    ref = O.State.create(O.Params(Lx=Lx, Ly=Ly, m=1, **CFG), *_fields(Lx, Ly))
    ref.run(2)
    return Lx, Ly, ref


@pytest.mark.parametrize("tuning", [None, "1,8,2,0,32", "1,16,2,2,32"])
def test_tall(tall, tuning, monkeypatch):
    Lx, Ly, ref = tall
    if tuning:
        monkeypatch.setenv("HLBM_TUNING", tuning)
    else:
        monkeypatch.delenv("HLBM_TUNING", raising=False)
    lat = lbm.Lattice(lbm.LbmParams(Lx=Lx, Ly=Ly, fd_substeps=-1, precision=lbm.LBM_F64, **CFG))
    lat.init_fields(*_fields(Lx, Ly)).step(2)
    gn, gphi, gu = lat.moments()
    rn, ru = ref.moments()
    assert np.max(np.abs(gphi - ref.phi)) <= 1e-11
    assert np.max(np.abs(gu - ru)) <= 1e-12
    assert np.max(np.abs(gn - rn)) <= 1e-11
    lat.close()


def test_small_tile_collide_is_refused(monkeypatch):
    monkeypatch.setenv("HLBM_TUNING", "1,32,2,8,32")
    with pytest.raises(Exception, match="HLBM_TUNING"):
        lbm.Lattice(lbm.LbmParams(Lx=3, Ly=524281, fd_substeps=-1, precision=lbm.LBM_F64, **CFG))
