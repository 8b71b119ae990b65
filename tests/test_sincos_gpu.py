"""The sine and cosine of exp(psi) themselves, against double precision.

Bound up to 65536 rad, absolute: two roundings of the reduced phase (2^-25 each,
it is below 1), one of the result (2^-25), the polynomials' fit (2^-27.9) and the
roundings of their last product (below 2^-27): 1.7 x 2^-24. Beyond, the library's
bits."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = 1.7 * 2.0 ** -24


@pytest.fixture(scope="module")
def sincos():
    from paper_2503_20146_gb300 import _build as B
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "sincos_probe.cu")
    lib = os.path.join(B.OBJDIR, "sincos_probe.so")
    os.makedirs(B.OBJDIR, exist_ok=True)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-I", os.path.join(B.ROOT, "include"), "-I", B.CSRC, "-shared", src,
                    "-o", lib], check=True)
    probe = ctypes.CDLL(lib)

    def run(y, library=False):
        d_y = torch.from_numpy(y).cuda()
        out = torch.zeros((2, len(y)), device="cuda")
        torch.cuda.synchronize()
        assert probe.probe_sincos(ctypes.c_void_p(d_y.data_ptr()), ctypes.c_void_p(out.data_ptr()), len(y), int(library)) == 0
        return out.cpu().numpy()

    return run


@pytest.mark.parametrize("reach", [math.pi / 4, 3.2, 50.0, 4000.0, 65536.0])
def test_absolute_error(sincos, reach):
    rng = np.random.default_rng(int(reach))
    y = rng.uniform(-reach, reach, 1 << 20).astype(np.float32)
    # the edges of the quadrants and the zeros, one number to either side, and the ends of the range
    edges = (np.arange(-64, 65) * (math.pi / 4)).astype(np.float32)
    edges = np.concatenate([edges, np.nextafter(edges, np.float32(1e9)), np.nextafter(edges, np.float32(-1e9))])
    y = np.concatenate([y, edges, np.float32([0.0, -0.0, reach, -reach])]).astype(np.float32)
    s, c = sincos(y)
    y64 = y.astype(np.float64)
    es, ec = s - np.sin(y64), c - np.cos(y64)
    assert max(np.abs(es).max(), np.abs(ec).max()) <= TOL
    gain = np.mean(s.astype(np.float64) ** 2 + c.astype(np.float64) ** 2) - 1.0
    assert abs(gain) <= 2.0 ** -28  # the modulus is right on average


def test_library_beyond(sincos):
    y = np.float32([65537.0, -65537.0, 1e6, -3e7, 1e20, -3e38, np.nextafter(np.float32(65536), np.float32(1e9))])
    assert np.array_equal(sincos(y), sincos(y, library=True))
    assert np.isnan(sincos(np.float32([np.inf, -np.inf, np.nan]))).all()
