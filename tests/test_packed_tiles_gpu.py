"""What the tiles of the packed residual pass read: positions 0 and nx/2 of a
packed row belong to the CTAs of bins 0 and nx/2, which write them in the same
launch, so a tile must not depend on them. The tiles run alone, once over zeros
and once over NaN in those positions: every other position the same to the bit,
the loss the same up to the order of its double-precision sum, and positions 0
and nx/2 left as they were."""
import ctypes
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe():
    from paper_2503_20146_gb300 import _build as B
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "packed_probe.cu")
    lib = os.path.join(B.OBJDIR, "packed_probe.so")
    os.makedirs(B.OBJDIR, exist_ok=True)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-I", os.path.join(B.ROOT, "include"), "-I", B.CSRC, "-shared", src,
                    "-o", lib], check=True)
    return ctypes.CDLL(lib)


@pytest.mark.parametrize("nproj,nx", [(1, 16), (1, 64), (3, 96)])
def test_tiles_do_not_depend_on_the_edge_bins(probe, nproj, nx):
    n = 64
    g = torch.Generator(device="cuda").manual_seed(nx)
    rnd = lambda *s: torch.randn(*s, 2, device="cuda", generator=g).view(torch.float32)  # noqa: E731
    field = torch.view_as_complex(rnd(nproj, n, nx).contiguous())
    yhat = torch.view_as_complex(rnd(nproj, n, nx).contiguous())
    ix, iy = torch.rand(nx, device="cuda", generator=g), torch.rand(n, device="cuda", generator=g)
    tw = torch.zeros(2 * n, dtype=torch.complex64, device="cuda")
    out = []
    for fill in (0.0, float("nan")):
        x = field.clone()
        x[:, 0::2, 0] = x[:, 0::2, nx // 2] = complex(fill, fill)  # packed rows sit on the even rows
        acc = torch.zeros((nproj, 8), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ptr = lambda v: ctypes.c_void_p(v.data_ptr())  # noqa: E731
        assert probe.probe_packed_tiles(ptr(x), ptr(yhat), ptr(ix), ptr(iy), ptr(tw), ptr(acc), nproj, nx) == 0
        edge = torch.view_as_real(x[:, 0::2][:, :, [0, nx // 2]])
        assert bool(torch.isnan(edge).all()) if fill != 0.0 else bool((edge == 0.0).all())
        x[:, 0::2, 0] = x[:, 0::2, nx // 2] = 0.0
        out.append((x, acc))
    assert torch.equal(out[0][0], out[1][0])
    assert bool(torch.isfinite(out[1][1]).all()) and float(out[0][1][:, 0].min()) > 0.0
    assert torch.allclose(out[0][1], out[1][1], rtol=1e-12, atol=0.0)
