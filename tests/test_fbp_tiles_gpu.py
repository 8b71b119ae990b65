"""The tile form of the back projection against the FP64 oracle, at the edges of
its rule and of its tiles: rows around the 64- and 128-slice blocks, odd angle
counts, angles outside [0, pi), the axes and diagonals, an output that starts
off a 16-byte boundary, more angles than one launch carries.

Tolerance: a position is exact to 2^-20 columns, which moves an interpolated
value by at most 2^-20 |q1 - q0| <= 2^-19 max|q|, about 7e-6 of the rms of white
noise (max about 3.5 rms); filter and sums in FP32 stay below 1e-6."""
import math

import numpy as np
import pytest

from oracle import fbp_oracle as F
from paper_2503_20146_gb300 import synth as S

from _cases import rel_l2

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def pwf():
    from paper_2503_20146_gb300 import _build
    _build.build()
    from paper_2503_20146_gb300 import pwf as P
    P.load()
    return P


def random_psi(n_angles, ny, nx, seed):
    rng = np.random.default_rng(seed)
    return (rng.standard_normal((n_angles, ny, nx)) + 1j * rng.standard_normal((n_angles, ny, nx))).astype(np.complex64)


def check_rows(vol, psi, angles, rows):
    ref = F.fbp_volume(psi[:, rows, :].astype(np.complex128), angles, S.WAVELENGTH_20KEV_M, S.PIXEL_M)
    got = vol[rows].cpu().numpy()
    assert rel_l2(got, ref) < TOL, rel_l2(got, ref)


@pytest.mark.parametrize("n_angles,ny,nx", [(1, 64, 128), (7, 32, 128), (12, 31, 128), (5, 63, 192), (6, 65, 96),
                                           (9, 127, 64), (4, 129, 128), (300, 40, 128), (3, 513, 48), (2, 33, 1024)])
def test_tile_form_matches_oracle(pwf, n_angles, ny, nx):
    psi = random_psi(n_angles, ny, nx, 31 * ny + nx)
    angles = np.random.default_rng(ny).uniform(-math.pi, 2.0 * math.pi, n_angles)
    fixed = [0.0, math.pi / 2, math.pi / 4, 3 * math.pi / 4, -math.pi, math.atan(0.5)]
    angles[:min(n_angles, 6)] = fixed[:min(n_angles, 6)]
    vol = pwf.pwf_fbp(torch.from_numpy(psi).cuda(), angles, S.WAVELENGTH_20KEV_M, S.PIXEL_M)
    check_rows(vol, psi, angles, sorted({0, 1, ny // 2, min(ny - 1, 64), ny - 1}))


def test_tile_form_output_off_a_16_byte_boundary_and_untouched_neighbours(pwf):
    n_angles, ny, nx = 8, 70, 128
    psi = random_psi(n_angles, ny, nx, 5)
    angles = S.tomo_angles(n_angles)
    buf = torch.full((ny * nx * nx + 2,), 7.0 + 1.0j, dtype=torch.complex64, device="cuda")
    vol = buf[1:-1].view(ny, nx, nx)
    assert vol.data_ptr() % 16 == 8
    pwf.pwf_fbp(torch.from_numpy(psi).cuda(), angles, S.WAVELENGTH_20KEV_M, S.PIXEL_M, vol=vol)
    check_rows(vol, psi, angles, [0, 63, 64, ny - 1])
    assert complex(buf[0]) == 7.0 + 1.0j and complex(buf[-1]) == 7.0 + 1.0j


@pytest.mark.parametrize("ny", [8, 64])
def test_an_angle_that_is_not_finite_gives_nan(pwf, ny):
    psi = torch.from_numpy(random_psi(4, ny, 128, 2)).cuda()
    vol = pwf.pwf_fbp(psi, [0.1, float("nan"), 1.0, 2.0], S.WAVELENGTH_20KEV_M, S.PIXEL_M)
    assert bool(torch.isnan(vol.real).all()) and bool(torch.isnan(vol.imag).all())
