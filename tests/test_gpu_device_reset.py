"""Nothing that the library keeps on the device or in pinned memory outlives the
lattices: a program may end its CUDA context between two of them."""
import os
import subprocess
import sys

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

_PROGRAM = """
import ctypes, sys
sys.path.insert(0, {root!r})
from paper_1908_05396_gb300 import build, clbm, workloads as wl
build.build()

def run(n):
    lats = [clbm.Lattice(16, 16, 16, face=wl.CAVITY_FACES, K=0.02, n=0.7, U_lid=(0.05, 0.0, 0.0),
                         dtype=d, check_interval=10) for d in ("f64", "f32", "f16s", "f16r")[:n]]
    out = []
    for lat in lats:
        lat.step(20)
        out.append((lat.residual()[0], lat.mass()))
    for lat in lats:
        lat.close()
    return out

a = run(4)
with open("/proc/self/maps") as f:
    name = next(l.split()[-1] for l in f if "libcudart" in l)
assert ctypes.CDLL(name).cudaDeviceReset() == 0
for x, y in zip(run(4), a):     # (sums of a few blocks' FP64 parts, in any order)
    assert abs(x[0] - y[0]) <= 1e-12 * y[0] and abs(x[1] - y[1]) <= 1e-12 * y[1]
"""


def test_lattices_after_a_device_reset():
    r = subprocess.run([sys.executable, "-c", _PROGRAM.format(root=ROOT)], capture_output=True,
                       text=True, timeout=300, env=dict(os.environ))
    assert r.returncode == 0, r.stderr[-2000:]
