"""Edges of the float32 kernels' dispatch rules (``-m gpu``)."""
import numpy as np
import pytest

from paper_2406_07366_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _B():
    import paper_2406_07366_gb300 as B
    return B


def _parts(B, f, **kw):
    bs = B.BiotSavart(B.make_params(f.L, **kw), f.offsets, f.closing)
    p = bs.parts(torch.from_numpy(f.nodes).cuda())
    torch.cuda.synchronize()
    bs.close()
    return p.cpu().numpy()


@pytest.mark.parametrize("rc_over_L", [0.30, 0.24, 0.21, 0.11, 0.06])
@pytest.mark.parametrize("sizes", [(7, 33), (64,), (5, 5, 5, 5), (101, 16)])
def test_short_range_of_node_pairs(sizes, rc_over_L):
    """Node pairs per warp where the grid has 2 (m + 2) cells per axis (rc below
    a quarter of the box at two cells per cut-off), single nodes on coarser
    grids: odd node counts, pairs that span two filaments or distant cells,
    curves across the box boundary.  Against the float64 form at float32's
    1e-5 (rms), the tolerance of the mixed-precision parity tests."""
    B = _B()
    rng = np.random.default_rng(len(sizes))
    curves = []
    for k, n in enumerate(sizes):
        th = 2 * np.pi * np.arange(n) / n
        c = np.array([0.05, 6.2, 3.0]) * (k % 2) + rng.uniform(0, 6, 3) * (1 - k % 2)
        curves.append(c + np.stack([0.4 * np.cos(th), 0.3 * np.sin(th), 0.2 * np.sin(2 * th)], 1) * (0.3 + 0.02 * n))
    f = W._pack(curves, 2 * np.pi)
    rc = rc_over_L * 2 * np.pi
    kw = dict(M=32, Q=2, w=8, alpha=3.5 / rc, rc=rc)
    a = _parts(B, f, precision=B.BS_MIXED, **kw)[1]
    b = _parts(B, f, precision=B.BS_FP64, **kw)[1]
    assert np.sqrt(((a - b) ** 2).mean()) <= 1e-5 * np.sqrt((b ** 2).mean())
