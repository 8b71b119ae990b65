"""Shapes the plan-time tuner offers: each costs every plan its preparation and
timing, so the single-buffered tiles of one column per thread ("C8s"), which win
only from length 1024 on, are offered there only."""
import re

import pytest

from paper_2503_20146_gb300 import synth as S

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

W = S.WORKLOADS["blob512_iotf"]


@pytest.fixture(scope="module")
def pwf():
    from paper_2503_20146_gb300 import _build
    _build.build()
    from paper_2503_20146_gb300 import pwf as P
    P.load()
    return P


@pytest.mark.parametrize("ny,offered", [(64, False), (96, False), (128, False), (256, False), (512, False), (768, False),
                                        (1024, True), (1536, True)])
def test_single_buffered_tiles_only_where_they_win(pwf, ny, offered):
    desc = pwf.PlanDesc(1, ny, 64, W.pixel_m, W.wavelength_m, W.L1_m, W.L2_m, W.xcoh_m, W.ycoh_m, W.gamma, W.alpha.real,
                        W.alpha.imag, W.eta, 0)
    with pwf.Plan(desc) as plan:
        text = pwf.pwf_plan_describe(plan.handle)
    shapes = re.search(r" col_q=[^\[]*\[([^\]]*)\]", text).group(1).split(",")
    names = [s.split(":")[0] for s in shapes]
    assert ("C8s" in names) == offered and "C4s" not in names, names
