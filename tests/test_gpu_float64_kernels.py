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


@pytest.mark.parametrize("n", [4, 5, 31, 32, 33, 256, 257, 1828, 1829])
def test_float64_cubic_fit_at_the_edges_of_its_size_rule(n):
    """Parallel cyclic reduction up to 1828 nodes per filament, the serial
    sweeps beyond: 1e-12 of the box and 1e-11 of the largest charge against the
    oracle's collocation, as for the quintic fit."""
    B, f = _B(), _uneven_ring(n, n) if n > 5 else W.ring(R=0.3, N=n)
    p = B.make_params(f.L, M=32, Q=2, w=8, precision=B.BS_FP64)
    bs = B.BiotSavart(p, f.offsets, f.closing)
    v = bs.velocity(torch.from_numpy(f.nodes).cuda())
    qX, qq = bs.quadrature(torch.from_numpy(f.nodes).cuda())
    torch.cuda.synchronize()
    bs.close()
    assert torch.isfinite(v).all()
    g = oracle.geometry(f.nodes, f.offsets, f.closing, f.L, 4, 2)
    d = qX.cpu().numpy() - g.qX
    d -= f.L * np.round(d / f.L)
    assert np.abs(d).max() < 1e-12 * f.L.max()
    assert np.abs(qq.cpu().numpy() - g.qq).max() < 1e-11 * np.abs(g.qq).max()


def test_energy_line_on_both_sides_of_its_size_rule():
    """A ring of 3200 nodes (a CTA per filament) and one of 3201 (a warp):
    between them the local terms' O(l^2) error, 4e-6 here, changes by 6e-4 of
    itself, 3e-9 of the energy."""
    B = _B()
    E = []
    for n in (3200, 3201):
        f = W.ring(N=n)
        p = B.make_params(f.L, M=32, Q=2, w=8, precision=B.BS_FP64, flags=B.BS_WANT_PSI)
        bs = B.BiotSavart(p, f.offsets, f.closing)
        E.append(bs.energy(torch.from_numpy(f.nodes).cuda()))
        bs.close()
    assert abs(E[0] - E[1]) < 1e-8 * abs(E[0])


@pytest.mark.parametrize("sigma", [1.25, 1.5, 2.0])
@pytest.mark.parametrize("w", [2, 4, 6, 8, 10, 12, 14, 16])
def test_float64_kernel_polynomials_equal_the_kernel(w, sigma):
    """The long-range part with polynomial kernel weights (the default path,
    every column block shape the sizes give) against the full-transform path,
    which evaluates the kernel itself.  Weight errors are below 3e-15 of the
    peak on either side; a part is a sum of such terms: 1e-12 of its largest value."""
    B, f = _B(), W.ellipses(3, 40, seed=11)
    nodes = torch.from_numpy(f.nodes).cuda()
    parts = []
    for flags in (0, B.BS_FFT_CUFFT):
        p = B.make_params(f.L, M=33, Q=2, w=w, sigma=sigma, precision=B.BS_FP64, flags=flags)
        bs = B.BiotSavart(p, f.offsets, f.closing)
        parts.append(bs.parts(nodes)[2].clone())
        torch.cuda.synchronize()
        bs.close()
    assert float((parts[0] - parts[1]).abs().max()) < 1e-12 * float(parts[1].abs().max())


@pytest.mark.parametrize("local_frac", [0.0, 0.1])
@pytest.mark.parametrize("order,total", [(4, 4864), (4, 4865), (6, 4865)])
def test_float64_node_terms_by_lanes_equal_a_thread_per_node(order, total, local_frac):
    """Up to 4864 nodes 8 lanes share a node's quadrature points, beyond it a
    thread takes the node.  The local and self terms depend on the node's own
    filament alone, so a 65-node curve has the same ones by itself and beside
    others: sums of at most 2 (2 + 4) Q terms in another order, 1e-12 of the
    largest (the float64 parity tolerance)."""
    B, a = _B(), _uneven_ring(65, 7)
    rest = total - 65 - 64 * 73
    X = [a.nodes] + [_uneven_ring(64, k).nodes for k in range(73)] + [_uneven_ring(rest, 99).nodes]
    f = W._pack(X, a.L)
    assert len(f.nodes) == total
    out = []
    for s in (a, f):
        p = B.make_params(s.L, M=32, Q=3, order=order, w=8, precision=B.BS_FP64, alpha=4.0, rc=1.5,
                          flags=B.BS_WANT_PSI, local_frac=local_frac)
        bs = B.BiotSavart(p, s.offsets, s.closing)
        v, psi = bs.parts(torch.from_numpy(s.nodes).cuda(), want_psi=True)
        torch.cuda.synchronize()
        bs.close()
        out.append([x[k, :65].cpu().numpy() for x in (v, psi) for k in (0, 3)])
    for x, y in zip(*out):
        assert np.abs(x - y).max() < 1e-12 * np.abs(x).max()


def _erfc_g(x):
    """erfc(x) and g(x) = erfc(x) + 2/sqrt(pi) x exp(-x^2) of a Decimal, at the context's precision."""
    from decimal import Decimal
    c = 2 / Decimal("3.14159265358979323846264338327950288419716939937510582097494459230781640628620899862803").sqrt()
    term, s, n = x, x, 0
    while abs(term) > Decimal(10) ** -70:
        n += 1
        term *= -x * x / n
        s += term / (2 * n + 1)
    e = 1 - c * s
    return e, e + c * x * (-x * x).exp()


@pytest.mark.parametrize("alpha", [0.25, 1.0, 1.5, 2.0])
def test_float64_pair_functions_relative_to_themselves(alpha):
    """Two lines at right angles, two lengths apart, with their reverses out of
    reach: at a node of one line psi points along the other line and the
    velocity's part across both comes from it alone, from separations r of the
    node's distance and a little more.  So each node shows erfc(alpha r) and
    g(alpha r) relative to themselves, up to alpha r = 8.  Coordinates are
    exact in binary but for the quadrature points along the lines; three
    roundings of r are amplified by the functions' (x^2 2 relative), the rest
    is a dozen roundings: (16 x^2 + 32) 2^-53."""
    from decimal import Decimal, localcontext
    B, n, rc = _B(), 32, 4.0
    L = np.full(3, 16.0)
    t = 0.5 * np.arange(n)

    def line(axis, *at):
        X = np.empty((n, 3))
        X[:, axis] = t
        X[:, [k for k in range(3) if k != axis]] = at
        return X

    a, b = line(2, 0.5, 8.5), line(1, 2.5, 8.25)              # along z; along y, 2 away in x
    back_a, back_b = line(2, 8.5, 8.5)[::-1], line(1, 10.5, 8.25)[::-1]
    f = W._pack([a, b, back_a, back_b], L, closing=[[0, 0, 1], [0, 1, 0], [0, 0, -1], [0, -1, 0]])
    p = B.make_params(L, M=32, Q=3, w=8, alpha=alpha, rc=rc, flags=B.BS_WANT_PSI, precision=B.BS_FP64)
    bs = B.BiotSavart(p, f.offsets, f.closing)
    nodes = torch.from_numpy(f.nodes).cuda()
    v, psi = bs.parts(nodes, want_psi=True)
    qX, qq = bs.quadrature(nodes)
    bs.status()
    bs.close()
    vz, py = v[1][:n, 2].cpu().numpy(), psi[1][:n, 1].cpu().numpy()
    Y, q = qX.cpu().numpy()[3 * n:6 * n], qq.cpu().numpy()[3 * n:6 * n, 1]
    seen = 0
    with localcontext() as ctx:
        ctx.prec = 110
        for j in range(n):
            ev = ep = Decimal(0)
            dz = Decimal(8.25) - Decimal(float(a[j, 2]))
            for y, c in zip(Y[:, 1], q):
                dy = Decimal(float(y)) - Decimal(8.5)
                r2 = 4 + dy * dy + dz * dz
                if r2 >= 16:
                    continue
                r = r2.sqrt()
                e, g = _erfc_g(Decimal(alpha) * r)
                ev += 2 * Decimal(float(c)) * g / (r2 * r)    # (r x q)_z = r_x q_y
                ep += Decimal(float(c)) * e / r
            if ep == 0:
                continue
            seen += 1
            pre = Decimal(p.kappa / (4 * math.pi))
            x2 = alpha ** 2 * (4 + float(dz) ** 2)
            tol = (16 * x2 + 32) * 2.0 ** -53
            assert abs(Decimal(float(vz[j])) / (pre * ev) - 1) < tol, (j, math.sqrt(x2))
            assert abs(Decimal(float(py[j])) / (pre * ep) - 1) < tol, (j, math.sqrt(x2))
    assert seen >= 12
