"""Shared memory limits of the launches (``-m gpu``)."""
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


def _ring(n, L=2 * math.pi):
    th = 2 * math.pi * np.arange(n) / n
    return W._pack([np.stack([np.cos(th), np.sin(th), 0.3 * np.sin(2 * th)], 1) + L / 2], L)


# The fits hold 9 float32 values (mixed, cubic), 14 float64 (cubic) or 32 float64
# (quintic) a node beside a few hundred static bytes; 48 KB is what a launch gets
# without asking for more.
@pytest.mark.parametrize("prec,order,n", [("mixed", 4, 1364), ("mixed", 4, 1365), ("mixed", 4, 1366),
                                          ("fp64", 4, 437), ("fp64", 4, 438), ("fp64", 4, 439), ("mixed", 6, 191),
                                          ("mixed", 6, 192), ("fp64", 6, 191), ("fp64", 6, 192), ("fp64", 6, 193)])
def test_fits_whose_buffers_nearly_fill_48_kb(prec, order, n):
    """Points and charges against the oracle's collocation: 1e-12 of the box and
    1e-11 of the largest charge in float64, 2.4e-6 of the longest chord and of
    the largest charge in float32 (the bounds of the other fit tests)."""
    B, f = _B(), _ring(n)
    p = B.make_params(f.L, M=32, Q=2, w=8, order=order, precision=B.BS_FP64 if prec == "fp64" else B.BS_MIXED)
    bs = B.BiotSavart(p, f.offsets, f.closing)
    nodes = torch.from_numpy(f.nodes).cuda()
    v = bs.velocity(nodes)
    qX, qq = bs.quadrature(nodes)
    bs.status()
    bs.close()
    assert torch.isfinite(v).all()
    g = oracle.geometry(f.nodes, f.offsets, f.closing, f.L, order, 2)
    chord = np.linalg.norm(np.diff(f.nodes, axis=0), axis=1).max()
    d = qX.cpu().numpy() - g.qX
    d -= f.L * np.round(d / f.L)
    assert np.abs(d).max() < (1e-12 * f.L.max() if prec == "fp64" else 2.4e-6 * chord)
    assert np.abs(qq.cpu().numpy() - g.qq).max() < (1e-11 if prec == "fp64" else 2.4e-6) * np.abs(g.qq).max()


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("order,n0,n", [(4, 764, 765), (4, 764, 768), (6, 190, 191), (6, 190, 192)])
def test_energies_whose_buffers_nearly_fill_48_kb(prec, order, n0, n):
    """The energy of a curve of n nodes against n0, which stays clear of 48 KB:
    discretisation errors are below 1e-3 here and go with the square of the
    spacing, which differs by at most 2 per cent: 4e-5 of the energy."""
    B = _B()
    E = []
    for k in (n0, n):
        f = _ring(k)
        p = B.make_params(f.L, M=32, Q=2, w=8, order=order, flags=B.BS_WANT_PSI,
                          precision=B.BS_FP64 if prec == "fp64" else B.BS_MIXED)
        bs = B.BiotSavart(p, f.offsets, f.closing)
        E.append(bs.energy(torch.from_numpy(f.nodes).cuda()))
        bs.close()
    assert abs(E[1] - E[0]) < 4e-5 * abs(E[0])


@pytest.mark.parametrize("n", [1364, 1365])
def test_staged_batch_whose_fit_nearly_fills_48_kb(n):
    """One mixed member with a filament of n nodes, staged: its velocity against
    its single context (1e-6, the tolerance of the batch tests)."""
    B, f = _B(), _ring(n)
    p = B.make_params(f.L, M=32, Q=2, w=8, precision=B.BS_MIXED)
    p.flags |= B.BS_BATCH_STAGED
    nodes = torch.from_numpy(f.nodes).cuda()
    bt = B.BiotSavartBatch([p], [f], stream=torch.cuda.Stream())
    torch.cuda.synchronize()
    got = bt.velocity(nodes)
    bt.status()
    assert tuple(int(x) for x in bt.staged) == (1,)
    bt.close()
    bs = B.BiotSavart(p, f.offsets, f.closing)
    ref = bs.velocity(nodes)
    bs.status()
    bs.close()
    assert float((got - ref).abs().max()) < 1e-6 * float(ref.abs().max())


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_contexts_of_different_sizes_in_several_threads(prec):
    """A kernel's shared memory limit belongs to the function, not to a context:
    contexts whose launches need different amounts (grids of 48 to 192 points,
    filaments of 64 to 1500 nodes), each driven by a thread of its own, must not
    lower it for one another.  Every evaluation equals the context's first one
    (float32 atomics reorder the mixed sums: 1e-6; float64 1e-12)."""
    import threading
    B = _B()
    out, err = {}, []

    def drive(k, M, n):
        try:
            f = _ring(n)
            s = torch.cuda.Stream()
            p = B.make_params(f.L, M=M, Q=2, w=8, precision=B.BS_FP64 if prec == "fp64" else B.BS_MIXED)
            bs = B.BiotSavart(p, f.offsets, f.closing, stream=s)
            nodes = torch.from_numpy(f.nodes).cuda()
            v = [torch.empty_like(nodes) for _ in range(2)]
            torch.cuda.synchronize()
            bs.velocity(nodes, v[0])
            ready.wait(60)
            for _ in range(400):
                bs.velocity(nodes, v[1])
            bs.status()
            out[k] = float((v[1] - v[0]).abs().max() / v[0].abs().max())
            bs.close()
        except Exception as e:  # noqa: BLE001 (shown by the main thread)
            err.append(repr(e))
            ready.abort()

    sizes = [(32, 64), (64, 400), (96, 1000), (128, 1500)]
    ready = threading.Barrier(len(sizes))
    threads = [threading.Thread(target=drive, args=(k, *s)) for k, s in enumerate(sizes)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not err, err
    assert len(out) == len(sizes) and max(out.values()) < (1e-6 if prec == "mixed" else 1e-12), out
