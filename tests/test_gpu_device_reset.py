"""The calls without a context of the library's own go on after a device reset.

Other code of the process may reset the device; everything allocated on it is
gone then, the library's scratch pool too.  Interpolation, resistivity and
sub-domain solves, which keep no handle between calls, must work as before.  In
a child process, which only ends its own context by the reset.
"""
import subprocess
import sys
from pathlib import Path

import pytest

from paper_1603_09311_gb300 import build as B

pytestmark = pytest.mark.gpu

CHILD = """
import ctypes, sys
import numpy as np
import torch
sys.path.insert(0, sys.argv[1])
from paper_1603_09311_gb300 import inputs as I, sdd

def calls():
    s = np.arange(12.0)
    v = np.sin(s)[:, None]
    a, e = sdd.sdd_interpolate(s, v, 0.1 * np.abs(v), np.array([0.5, 3.3, 10.9]), 1)
    nodes, edge = I.rect_grid(0.0, 0.9, 0.0, 0.9, 20, 20)
    u, _ = sdd.sdd_rbffd_solve(nodes, edge, np.where(edge == 1, 1.0 + nodes[:, 0], 0.0), np.full(400, 3.0), eps=5.0,
                               tol=1e-10)
    val = np.linspace(1.0, 2.0, 12).reshape(2, 3, 1, 2)
    r = sdd.sdd_apparent_from_values(val[..., 0] + 1j * val[..., 1], 0.01 * val, 0.02, [2.0])
    return [a, e, u] + [np.asarray(x) for x in (r.values() if isinstance(r, dict) else r)]

before = calls()
cudart = [l.split()[-1] for l in open("/proc/self/maps") if "libcudart" in l]
assert ctypes.CDLL(cudart[0]).cudaDeviceReset() == 0
for _ in range(2):
    assert all(np.array_equal(x, y, equal_nan=True) for x, y in zip(before, calls()))
print("same")
"""


def test_calls_after_a_device_reset():
    B.build()
    root = str(Path(__file__).resolve().parents[1])
    r = subprocess.run([sys.executable, "-c", CHILD, root], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split() == ["same"], r.stdout + r.stderr
