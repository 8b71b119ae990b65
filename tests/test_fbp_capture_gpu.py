"""pwf_fbp captured into a graph: it enqueues kernels only, so a replay gives the
bits of the ordinary call (tile form with four and two slices per lane, direct
form)."""
import numpy as np
import pytest

from paper_2503_20146_gb300 import synth as S

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pwf():
    from paper_2503_20146_gb300 import _build
    _build.build()
    from paper_2503_20146_gb300 import pwf as P
    P.load()
    return P


@pytest.mark.parametrize("n_angles,ny,nx", [(6, 70, 128), (5, 40, 256), (4, 3, 512)])
def test_under_capture(pwf, n_angles, ny, nx):
    rng = np.random.default_rng(ny)
    psi = (rng.standard_normal((n_angles, ny, nx)) + 1j * rng.standard_normal((n_angles, ny, nx))).astype(np.complex64)
    psi, ang = torch.from_numpy(psi).cuda(), S.tomo_angles(n_angles)
    ref = pwf.pwf_fbp(psi, ang, S.WAVELENGTH_20KEV_M, S.PIXEL_M)
    vol = torch.zeros_like(ref)
    ws = torch.empty(pwf.pwf_fbp_workspace_bytes(n_angles, ny, nx), dtype=torch.uint8, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        pwf.pwf_fbp(psi, ang, S.WAVELENGTH_20KEV_M, S.PIXEL_M, vol=vol, workspace=ws)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(vol, ref)
