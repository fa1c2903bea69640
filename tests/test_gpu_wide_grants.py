"""Shared memory of the wide-patch kernels is granted per kernel: an FP64 handle with larger patches
between two FP32 handles must not stand in for the second one's grant. In a process of its own, since
any earlier grant would hide the order."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

_CODE = """
import numpy as np
from paper_1504_07028_gb300 import binding as B
for M, prec, dt in ((3, "fp32", np.float32), (5, "fp64", np.float64), (5, "fp32", np.float32)):
    s = B.Solver(B.make_params(14, 19, %d, M=M, sigma=2.0, precision=prec))
    s.set_probs(np.full((%d, 14, 19), 1.0 / %d, dt))
    s.solve(3, trace_every=2)
    assert np.isfinite(s.get_z()).all()
    s.close()
"""


@pytest.mark.parametrize("K", [3, 7, 9, 17])
def test_grants_of_both_precisions(lib, K):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _CODE % (K, K, K)], cwd=root, timeout=300,
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
