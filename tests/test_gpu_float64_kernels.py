"""Edges of the float64 kernels' size rules (``-m gpu``), against the oracle."""
import math

import numpy as np
import pytest

import oracle
from paper_2406_07366_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _B():
    import paper_2406_07366_gb300 as B
    return B


def _uneven_ring(n, seed, L=2 * math.pi):
    """A closed curve of n nodes with chords that differ by up to a factor of about 3."""
    rng = np.random.default_rng(seed)
    th = np.cumsum(rng.uniform(0.5, 1.5, n))
    th *= 2 * math.pi / th[-1]
    X = np.stack([np.cos(th), np.sin(th), 0.3 * np.sin(2 * th)], 1) * (0.9 if n > 20 else 0.4) + L / 2
    return W._pack([X], L)


@pytest.mark.parametrize("n", [6, 7, 31, 32, 33, 255, 257, 800, 801])
def test_quintic_fit_at_the_edges_of_its_size_rule(n):
    """Parallel cyclic reduction (up to 800 nodes per filament, blocks of up
    to 256 threads) and the serial elimination beyond: points and charges
    against the oracle's B-spline collocation.  Both solve a well conditioned
    system (chord ratios below 3) in float64: 1e-12 of the box for points and
    1e-11 of the largest charge, as the other quintic tests."""
    B, f = _B(), _uneven_ring(n, n)
    p = B.make_params(f.L, M=32, Q=3, order=6, w=8, precision=B.BS_FP64)
    bs = B.BiotSavart(p, f.offsets, f.closing)
    qX, qq = bs.quadrature(torch.from_numpy(f.nodes).cuda())
    torch.cuda.synchronize()
    bs.close()
    g = oracle.geometry(f.nodes, f.offsets, f.closing, f.L, 6, 3)
    d = qX.cpu().numpy() - g.qX
    d -= f.L * np.round(d / f.L)
    assert np.abs(d).max() < 1e-12 * f.L.max()
    assert np.abs(qq.cpu().numpy() - g.qq).max() < 1e-11 * np.abs(g.qq).max()


@pytest.mark.parametrize("beta", [0.3, 3.5, 7.99, 8.01, 12.0])
def test_float64_short_range_over_the_table_and_beyond(beta):
    """The pair functions come from tables up to alpha r = 8 and from the
    library beyond; every r up to the cut-off against the oracle's brute
    force, 1e-12 relative to the largest velocity (the tolerance of the
    float64 parity tests)."""
    B, f = _B(), W.ellipses(6, 48, seed=3)
    rc = 2.0
    p = B.make_params(f.L, M=32, Q=2, w=8, precision=B.BS_FP64, alpha=beta / rc, rc=rc, flags=B.BS_WANT_PSI)
    bs = B.BiotSavart(p, f.offsets, f.closing)
    parts, psi = bs.parts(torch.from_numpy(f.nodes).cuda(), want_psi=True)
    torch.cuda.synchronize()
    bs.close()
    g = oracle.geometry(f.nodes, f.offsets, f.closing, f.L, 4, 2)
    v, ps = oracle.short_range(g, f.L, 1.0, p.alpha, p.rc)
    assert np.abs(parts[1].cpu().numpy() - v).max() < 1e-12 * np.abs(v).max()
    assert np.abs(psi[1].cpu().numpy() - ps).max() < 1e-12 * np.abs(ps).max()
