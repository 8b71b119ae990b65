"""pwf_fbp on two devices of one process. A kernel's limit of dynamic shared
memory belongs to the device it was set on, so the call has to set it on each.
Runs on CPU: a child process preloads a stand-in for the runtime calls with two
devices, which refuses a launch above the limit set on its device."""
import os
import shutil
import subprocess
import sys

import pytest

from paper_2503_20146_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))

CHILD = """
import ctypes, sys
from paper_2503_20146_gb300 import pwf
lib = pwf.load()
fake = ctypes.CDLL(None)
# tile form with four and two slices per lane, direct form, short rows and the longest
for n_angles, ny, nx in [(6, 70, 128), (5, 40, 256), (4, 3, 512), (3, 2, 1024), (300, 64, 1024), (2, 1, 16)]:
    need = lib.pwf_fbp_workspace_bytes(n_angles, ny, nx)
    angles = (ctypes.c_double * n_angles)(*[0.01 * k for k in range(n_angles)])
    for device in (0, 1, 0):
        fake.fake_set_device(device)
        before = fake.fake_launches()
        at = lambda k: ctypes.c_void_p(k << 40)  # nothing is launched: addresses that are only aligned
        status = lib.pwf_fbp(at(1), n_angles, ny, nx, angles, 1e-10, 1e-6, at(2), at(3), need, None)
        if status != 0 or fake.fake_launches() - before != 2 + (n_angles + 255) // 256:
            sys.exit(f"device {device}, {n_angles} x {ny} x {nx}: status {status}, "
                     f"{fake.fake_launches() - before} launches")
"""


def test_back_projection_on_a_second_device(tmp_path):
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        pytest.skip("no C compiler")
    _build.build()
    lib = str(tmp_path / "two_device_runtime.so")
    subprocess.run([cc, "-shared", "-fPIC", "-O1", os.path.join(HERE, "two_device_runtime.c"), "-o", lib], check=True)
    env = dict(os.environ, LD_PRELOAD=lib, PYTHONPATH=_build.ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, cwd=_build.ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
