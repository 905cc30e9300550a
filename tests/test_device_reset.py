"""Solves before and after the application resets the device (a child process: the reset ends its context)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import ctypes as C
import numpy as np
import oracle
from paper_2406_18001_gb300 import binding as B, inputs

B.lib()
rt = C.CDLL("libcudart.so.13")  # the one that the library has loaded
p = inputs.krr_dense(m=400, n=20, seed=3, dtype=np.float64)
want = oracle.bdcd_krr(p.A, p.y, oracle.kernel("rbf", gamma=0.5), 1e-2, 4, 12, seed=1)
for turn in range(3):
    al, _, _, _ = B.krr_solve(p.A, p.y, B.kernel("rbf", gamma=0.5), 1e-2, 4, 2, 12, seed=1, prec="fp64",
                              flags=B.FLAG_HOST_IO)
    assert np.linalg.norm(al - want) < 1e-10 * np.linalg.norm(want), turn
    assert rt.cudaDeviceReset() == 0
print("done")
"""


def test_solve_after_a_device_reset():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env={**os.environ, "PYTHONPATH": ROOT}, timeout=300,
                       capture_output=True, text=True)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout + r.stderr
