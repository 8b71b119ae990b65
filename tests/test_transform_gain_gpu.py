"""A transform followed by its inverse keeps the size of a field: with both
propagation distances 0 the coherent forward model is |exp(psi) t|^2, through two
filters of four transforms (two per axis) each. Rounded constants that are all a
little short of modulus 1 shrink every value alike, which shows in the mean
intensity of random fields, where ordinary rounding averages out.

Tolerance: half a unit of the last place, 2^-24, for a transform and its inverse
along one axis. The intensity sees four such pairs, squared: 8 x 2^-24. The
radix constants at their nearest FP32 values sum to -5.7e-7 (1536) and -6.7e-7
(1024, radix 32) over the eight."""
import numpy as np
import pytest

from paper_2503_20146_gb300 import synth as S

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

GAIN_TOL = 8.0 * 2.0 ** -24


@pytest.fixture(scope="module")
def pwf():
    from paper_2503_20146_gb300 import _build
    _build.build()
    from paper_2503_20146_gb300 import pwf as P
    P.load()
    return P


@pytest.mark.parametrize("n", [16, 32, 64, 96, 128, 256, 512, 768, 1024, 1536, 2048])
def test_mean_intensity_is_kept(pwf, n):
    w = S.WORKLOADS["blob128_coherent"]
    batch = max(1, (1 << 21) // (n * n))
    rng = np.random.default_rng(n)
    t = (rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))).astype(np.complex64)
    psi = (1j * rng.uniform(-3.0, 3.0, (batch, n, n))).astype(np.complex64)
    desc = pwf.PlanDesc(batch, n, n, w.pixel_m, w.wavelength_m, 0.0, 0.0, 0.0, 0.0, w.gamma, w.alpha.real, w.alpha.imag,
                        w.eta, pwf.FLAG_NO_TUNE)
    with pwf.Plan(desc) as plan:
        f = plan.forward(torch.from_numpy(psi).cuda(), torch.from_numpy(t).cuda())
    ref = float(np.mean(np.abs(t.astype(np.complex128)) ** 2))
    gain = float(f.double().mean()) / ref - 1.0
    assert abs(gain) <= GAIN_TOL, gain
