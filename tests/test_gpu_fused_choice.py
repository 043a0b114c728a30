"""GPU: the autotuner takes the one-launch 2D step only where it clearly beats the
two kernels: under 0.85 of the sum of their times as it prints them (near that line a
graph of the two kernels is faster than the timed launches tell) and, unless under
0.6, where a run of one step takes at most 1.12 of theirs."""
import re

import pytest

from paper_0902_3921_gb300 import lbm

pytestmark = pytest.mark.gpu


# far below the line, around it (m = 4 and m = 1), and beyond; sides that no other
# test uses, so that the tuner runs
@pytest.mark.parametrize("side,Gamma", [(62, 0.5), (250, 0.5), (438, 0.5), (474, 0.5), (506, 0.5), (522, 0.5),
                                        (506, 0.1), (690, 0.1), (866, 0.1)])
def test_choice_follows_the_printed_times(side, Gamma, monkeypatch, capfd):
    monkeypatch.delenv("HLBM_TUNING", raising=False)
    monkeypatch.setenv("HLBM_TUNE_VERBOSE", "1")
    kw = dict(a=-0.1, b=0.1, kappa=0.14, tau=1.0, N=0.3, Q=2.5, Gamma=Gamma)
    lat = lbm.Lattice(lbm.LbmParams(Lx=side, Ly=side, precision=lbm.LBM_F32DEV, **kw))
    tile = lbm.lbm_tuning(lat.handle)["fd_tile_width"]
    lat.close()
    err = capfd.readouterr().err
    lines = re.findall(r"fused step \d+x\d+ rows=\d+: ([0-9.]+) us \(separate kernels ([0-9.]+)\)", err)
    one = re.findall(r"one step \d+x\d+: fused kernel's halves ([0-9.]+) us, separate kernels ([0-9.]+)", err)
    assert len(lines) == 2 and lines[0][1] == lines[1][1]
    fused, separate = min(float(a) for a, _ in lines), float(lines[0][1])
    # printed to 0.1 us
    if fused > 0.85 * separate + 0.1:
        assert tile != 2 and not one
    if fused < 0.6 * separate - 0.1:
        assert tile == 2 and not one
    if one:
        halves, two = map(float, one[0])
        assert (tile == 2) == (halves <= 1.12 * two) or abs(halves - 1.12 * two) < 0.2
    assert (tile == 2) <= (fused <= 0.85 * separate + 0.1)
