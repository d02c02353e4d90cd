"""Contexts created after a device reset (``-m gpu``)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# A process of its own: a reset ends every context of the process.
CHILD = r"""
import ctypes, sys
import numpy as np
import paper_2406_07366_gb300 as B
from paper_2406_07366_gb300 import workloads as W

f = W.ellipses(3, 40, seed=2)

def velocity(prec):
    p = B.make_params(f.L, M=33, Q=2, w=8, precision=prec)     # 54 = 9 x 6 points: twiddles of every kind
    ctx = B.bs_create(p)
    B.bs_set_filaments(ctx, f.offsets, f.closing)
    v = np.empty_like(f.nodes)
    B.bs_compute_host(ctx, f.nodes, v)
    B.bs_status(ctx)
    B.bs_destroy(ctx)
    return v

before = [velocity(prec) for prec in (B.BS_FP64, B.BS_MIXED)]
path = [l.split()[-1] for l in open("/proc/self/maps") if "libcudart" in l][0]
assert ctypes.CDLL(path).cudaDeviceReset() == 0
for prec, v, tol in ((B.BS_FP64, before[0], 1e-12), (B.BS_MIXED, before[1], 1e-6)):
    w = velocity(prec)
    assert np.abs(w - v).max() < tol * np.abs(v).max(), (prec, np.abs(w - v).max() / np.abs(v).max())
"""


def test_new_contexts_after_a_device_reset_equal_the_earlier_ones():
    """The tables in device and constant memory are written again: float64 to
    1e-12, mixed to 1e-6 (float32 atomics reorder its sums)."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
