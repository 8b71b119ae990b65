"""exp(psi) in the forward model over the whole phase range: the polynomial sine
and cosine up to 65536 rad, the library routine beyond, both sides of the line
and of every quadrant. The object is float32 psi exactly, so the FP64 oracle
sees the same phases; forward tolerance 1e-5 as everywhere."""
import math

import numpy as np
import pytest

from oracle import pwf_oracle as O
from paper_2503_20146_gb300 import synth as S

from _cases import geometry, rel_l2

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pwf():
    from paper_2503_20146_gb300 import _build
    _build.build()
    from paper_2503_20146_gb300 import pwf as P
    P.load()
    return P


@pytest.mark.parametrize("centre", [0.0, 400.0, -65536.0, 65536.0, 3.0e5])
def test_forward_matches_oracle_at_any_phase(pwf, centre):
    n = 64
    w = S.WORKLOADS["blob512_iotf"]
    geom = geometry(w, n, n)
    rng = np.random.default_rng(3)
    phase = (centre + rng.uniform(-8.0, 8.0, (1, n, n))).astype(np.float32)
    phase[0, 0, :16] = np.float32(centre) + (np.arange(16) * math.pi / 4).astype(np.float32)
    psi = (rng.uniform(-1.0, 0.5, (1, n, n)).astype(np.float32) + 1j * phase).astype(np.complex64)
    t = S.diffuser(n, n, rng).astype(np.complex64)
    desc = pwf.PlanDesc(1, n, n, w.pixel_m, w.wavelength_m, w.L1_m, w.L2_m, w.xcoh_m, w.ycoh_m, w.gamma, w.alpha.real,
                        w.alpha.imag, w.eta)
    with pwf.Plan(desc) as plan:
        f = plan.forward(torch.from_numpy(psi).cuda(), torch.from_numpy(t).cuda()).cpu().numpy()[0]
    ref = O.intensity(psi[0].astype(np.complex128), t.astype(np.complex128), geom)
    assert rel_l2(f, ref) <= 1e-5, rel_l2(f, ref)


def test_infinite_phase_gives_nan(pwf):
    n = 32
    w = S.WORKLOADS["blob512_iotf"]
    psi = torch.zeros((1, n, n), dtype=torch.complex64, device="cuda")
    psi[0, 3, 4] = complex(0.0, float("inf"))
    t = torch.ones((n, n), dtype=torch.complex64, device="cuda")
    desc = pwf.PlanDesc(1, n, n, w.pixel_m, w.wavelength_m, w.L1_m, w.L2_m, w.xcoh_m, w.ycoh_m, w.gamma, w.alpha.real,
                        w.alpha.imag, w.eta)
    with pwf.Plan(desc) as plan:
        f = plan.forward(psi, t)
    assert bool(torch.isnan(f).all())
