"""Edges of the float32 kernels' dispatch rules (``-m gpu``)."""
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


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("sigma", [1.25, 1.5])
@pytest.mark.parametrize("M", [15, 31, 33, 43, 47, 63, 64, 85, 95, 97, 127, 130])
def test_boundary_passes_equal_full_transforms(M, sigma, prec):
    """The passes that start and end the transforms at the kept modes (grids
    with a factor 3 and K < n / 3, which sigma = 1.5 gives and 1.25 does not)
    and the general ones (powers of two, sigma = 1.25), with and without psi,
    against full cuFFT transforms.  Velocity and psi of the long range: 1e-12 of
    the largest value in float64; float32 transforms of 30 to 200 points, three
    axes both ways and sums of w^3 = 512 float32 terms, about 30 roundings of
    6e-8: 2e-6."""
    B, tol = _B(), 2e-6 if prec == "mixed" else 1e-12
    f = W.ellipses(3, 40, seed=M)
    nodes = torch.from_numpy(f.nodes).cuda()
    got = []
    for flags in (0, B.BS_WANT_PSI, B.BS_WANT_PSI | B.BS_FFT_CUFFT):
        p = B.make_params(f.L, M=M, Q=2, w=8, sigma=sigma, flags=flags, alpha=1.2, rc=3.0,
                          precision=B.BS_MIXED if prec == "mixed" else B.BS_FP64)
        bs = B.BiotSavart(p, f.offsets, f.closing)
        v = bs.parts(nodes, want_psi=bool(flags))
        got.append([x[2].clone() for x in (v if flags else (v,))])
        torch.cuda.synchronize()
        bs.close()
    ref = got[2]
    for x, r in ((got[0][0], ref[0]), (got[1][0], ref[0]), (got[1][1], ref[1])):
        assert float((x - r).abs().max()) < tol * float(r.abs().max())


@pytest.mark.parametrize("w", [2, 4, 6, 8, 10, 12, 14, 16])
@pytest.mark.parametrize("n", [37, 1219])
def test_gather_interpolation_by_a_warp_per_node(w, n):
    """The float32 gather of the streamfunction (a warp a node, one or four of
    them a block, one or more stages of planes) against the float64 context of
    the same parameters.  Float32 weights are within 2.2e-6 of their peak, three
    axes each at the spread and the gather, transforms and sums within 2e-6:
    3e-5 of the largest value."""
    B = _B()
    th = 2 * math.pi * np.arange(n) / n
    L = np.full(3, 2 * math.pi)
    X = np.stack([1.1 * np.cos(th), np.sin(th), 0.4 * np.cos(3 * th)], 1) + [0.2, 3.0, 6.1]
    f = W._pack([X], L)
    out = []
    for prec in (B.BS_FP64, B.BS_MIXED):
        p = B.make_params(f.L, M=32, Q=2, w=w, sigma=1.5, precision=prec, flags=B.BS_WANT_PSI)
        bs = B.BiotSavart(p, f.offsets, f.closing)
        out.append(bs.parts(torch.from_numpy(f.nodes).cuda(), want_psi=True)[1][2].cpu().numpy())
        bs.close()
    assert np.abs(out[1] - out[0]).max() < 3e-5 * np.abs(out[0]).max()


@pytest.mark.parametrize("closing", [0, 1])
@pytest.mark.parametrize("n,copies", [(4, 1), (31, 1), (33, 1), (256, 1), (257, 1), (600, 1), (40, 2433)])
def test_cubic_fit_by_a_block_per_filament(n, copies, closing):
    """A thread a node up to 2432 filaments, a warp beyond; closed curves and
    infinite ones.  Points and charges against the float64 fit of the oracle
    (its first filament): float32 chords and moments of a system with chord
    ratios below 3 are good to 20 roundings, 2.4e-6 of the longest chord for
    the points and of the largest charge."""
    B = _B()
    rng = np.random.default_rng(n)
    L = np.full(3, 2 * math.pi)
    th = np.cumsum(rng.uniform(0.5, 1.5, n))
    th *= 2 * math.pi / th[-1]
    X = np.stack([np.cos(th), np.sin(th), (th - th[0]) if closing else 0.3 * np.sin(2 * th)], 1) + L / 2
    # the closing offsets of a box sum to zero: each infinite curve with its reverse
    pair, close = ([X, X[::-1]], [[0, 0, 1], [0, 0, -1]]) if closing else ([X], [[0, 0, 0]])
    f = W._pack(pair * copies, L, closing=close * copies)
    p = B.make_params(f.L, M=32, Q=3, w=8, precision=B.BS_MIXED)
    bs = B.BiotSavart(p, f.offsets, f.closing)
    qX, qq = bs.quadrature(torch.from_numpy(f.nodes).cuda())
    torch.cuda.synchronize()
    bs.close()
    g = oracle.geometry(X, f.offsets[:2], f.closing[:1], f.L, 4, 3)
    shift = np.array([0, 0, closing * L[2]])
    chord = np.linalg.norm(np.diff(np.vstack([X, X[:1] + shift]), axis=0), axis=1).max()
    d = qX[:3 * n].cpu().numpy() - g.qX
    d -= f.L * np.round(d / f.L)
    assert np.abs(d).max() < 2.4e-6 * chord
    assert np.abs(qq[:3 * n].cpu().numpy() - g.qq).max() < 2.4e-6 * np.abs(g.qq).max()


@pytest.mark.parametrize("rc_over_L", [0.5, 0.4, 0.35])
def test_short_range_with_whole_axes_and_minimum_images(rc_over_L):
    """Cut-offs above a third of the box: every cell of an axis is a neighbour
    and separations wrap.  Velocity and streamfunction against the float64
    form at float32's 1e-5 (rms), as for the smaller cut-offs."""
    B, f = _B(), W.ellipses(7, 45, seed=5)
    rc = rc_over_L * 2 * math.pi
    out = []
    for prec in (B.BS_MIXED, B.BS_FP64):
        p = B.make_params(f.L, M=32, Q=2, w=8, alpha=3.5 / rc, rc=rc, flags=B.BS_WANT_PSI, precision=prec)
        bs = B.BiotSavart(p, f.offsets, f.closing)
        v, psi = bs.parts(torch.from_numpy(f.nodes).cuda(), want_psi=True)
        torch.cuda.synchronize()
        bs.close()
        out.append((v[1].cpu().numpy(), psi[1].cpu().numpy()))
    for a, b in zip(*out):
        assert np.sqrt(((a - b) ** 2).mean()) <= 1e-5 * np.sqrt((b ** 2).mean())


@pytest.mark.parametrize("M", [150, 299, 300])
def test_compiled_transforms_where_the_modes_pass_a_third(M):
    """sigma = 1.25 keeps K >= n / 3 of the modes on grids of 192 and 384 points,
    whose passes are compiled for their lengths: the whole transforms then end
    in a general last pass.  Long-range velocity and psi against full cuFFT
    transforms: 2e-6 as in the boundary-pass test, one more pass per axis at
    384 points: 3e-6."""
    B = _B()
    f = W.ellipses(3, 40, seed=M)
    nodes = torch.from_numpy(f.nodes).cuda()
    got = []
    for flags in (0, B.BS_WANT_PSI, B.BS_WANT_PSI | B.BS_FFT_CUFFT):
        p = B.make_params(f.L, M=M, Q=2, w=8, sigma=1.25, flags=flags, alpha=1.2, rc=3.0, precision=B.BS_MIXED)
        n, _ = B.bs_nufft_setup(p, want_table=False)
        assert tuple(n) == ((192,) * 3 if M == 150 else (384,) * 3) and 3 * ((M - 1) // 2) >= n[0]
        bs = B.BiotSavart(p, f.offsets, f.closing)
        v = bs.parts(nodes, want_psi=bool(flags))
        got.append([x[2].clone() for x in (v if flags else (v,))])
        torch.cuda.synchronize()
        bs.close()
    ref = got[2]
    for x, r in ((got[0][0], ref[0]), (got[1][0], ref[0]), (got[1][1], ref[1])):
        assert float((x - r).abs().max()) < 3e-6 * float(r.abs().max())


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("M", [35, 36, 39, 40, 41, 44, 47, 48])
def test_y_chunks_of_32_modes_with_tensor_copies(M, prec):
    """18 to 24 modes along z: the y pass takes them in one chunk of 32 and moves
    its rows with tensor copies where the count is even.  Long-range velocity
    and psi against full cuFFT transforms, bounds of the boundary-pass test."""
    B, tol = _B(), 2e-6 if prec == "mixed" else 1e-12
    f = W.ellipses(3, 40, seed=M)
    nodes = torch.from_numpy(f.nodes).cuda()
    got = []
    for flags in (0, B.BS_WANT_PSI, B.BS_WANT_PSI | B.BS_FFT_CUFFT):
        p = B.make_params(f.L, M=M, Q=2, w=8, flags=flags, alpha=1.2, rc=3.0,
                          precision=B.BS_MIXED if prec == "mixed" else B.BS_FP64)
        bs = B.BiotSavart(p, f.offsets, f.closing)
        v = bs.parts(nodes, want_psi=bool(flags))
        got.append([x[2].clone() for x in (v if flags else (v,))])
        torch.cuda.synchronize()
        bs.close()
    ref = got[2]
    for x, r in ((got[0][0], ref[0]), (got[1][0], ref[0]), (got[1][1], ref[1])):
        assert float((x - r).abs().max()) < tol * float(r.abs().max())
