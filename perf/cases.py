"""The work that users of this library have it do, as cases that can be timed and compared.

A case is a dict of plain values:

    call       velocity | energy (velocity, streamfunction and energy) | rk4 (one time step, graph replay)
               | host (velocity through host buffers) | batch (many configurations in one call)
    shape      ring | leapfrog | ellipses | tangle: the curves
    fil, per   filaments and nodes per filament (with ragged: per/2 .. 3 per/2 nodes each, drawn);
               a batch has fil configurations of per .. per_hi nodes each (log-uniform)
    precision  mixed | fp64
    M          resolved Fourier modes along the shortest side of the box (a batch: matched per member)
    Q, w, sigma, order, local_frac, deterministic   the method's options, as bs_params has them
    box        length of the y side over that of the others
"""
import math

import numpy as np
import torch

import paper_2406_07366_gb300 as B

KAPPA, CORE, DELTA, BETA, SIDE = 1.0, 1e-6, 0.25, 3.5, 2 * math.pi

_PLAIN = dict(call="velocity", shape="tangle", precision="mixed", fil=1, per=64, per_hi=0, ragged=False, M=32, Q=2,
              w=8, sigma=1.5, order=4, local_frac=0.0, deterministic=False, box=1.0)


def _case(name=None, **kw):
    c = dict(_PLAIN, **kw)
    return c if name is None else dict(name=name, **c)


def listed():
    return [
        # a single vortex ring: the smallest call, as in a convergence study or a first try; launches are all of it
        _case("ring 64", shape="ring", per=64, M=32),
        # one step of the conservation run of two leapfrogging rings: long runs of tiny steps in float64, with
        # quintic curves, three quadrature points and subdivided local segments (the paper's production setting)
        _case("leapfrog step", call="rk4", shape="leapfrog", precision="fp64", fil=2, per=32, M=17, Q=3, order=6,
              local_frac=0.1),
        # 40 random ellipses with their streamfunction and energy: the diagnostics of a small simulation
        _case("ellipses energy", call="energy", shape="ellipses", fil=40, per=64, M=64, Q=3),
        # the same curves' velocity in float64: reference runs and accuracy studies
        _case("ellipses fp64", shape="ellipses", precision="fp64", fil=40, per=64, M=64, Q=3),
        # filaments of unequal lengths (as reconnections leave them) in a box that is no cube, odd mode count, w = 6
        _case("ragged box", fil=73, per=127, ragged=True, M=97, Q=3, w=6, box=1.25),
        # an ordinary simulation's time step: 2e4 nodes, four velocity evaluations replayed as a graph
        _case("tangle 2e4 step", call="rk4", fil=200, per=100, M=128),
        # the 1e5-node tangle, one velocity evaluation in each precision
        _case("tangle 1e5", fil=1000, per=100, M=256),
        _case("tangle 1e5 fp64", precision="fp64", fil=1000, per=100, M=256),
        # a caller whose nodes live in host memory (pinned): copies in and out are part of the call
        _case("tangle 1e6 host", call="host", fil=5000, per=200, M=341),
        # the largest single evaluation: 4e6 nodes
        _case("tangle 4e6", fil=20000, per=200, M=512),
        # an ensemble of tangles of 1e3 to 1e5 nodes in one call, each with a grid of its own
        _case("batch 64", call="batch", fil=64, per=1000, per_hi=100000),
        # an ensemble of small tangles: many short members in one call
        _case("batch 256 small", call="batch", fil=256, per=250, per_hi=650),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    call = rng.choices(["velocity", "velocity fp64", "energy", "rk4", "host", "batch", "small"],
                       [6, 2, 2, 2, 1, 1, 2])[0]
    if call == "small":  # a few curves
        shape = rng.choice(["ring", "leapfrog", "ellipses"])
        fil = {"ring": 1, "leapfrog": 2, "ellipses": rng.randint(2, 48)}[shape]
        order = rng.choice([4, 4, 6])
        return _case(call=rng.choice(["velocity", "rk4", "energy"]), shape=shape, fil=fil, per=rng.randint(32, 160),
                     M=rng.randint(32, 72), Q=rng.choice([2, 3]), order=order,
                     precision=rng.choice(["mixed", "fp64"]), local_frac=rng.choice([0.0, 0.1]) if order == 6 else 0.0)
    if call == "batch":
        if rng.random() < 0.5:
            return _case(call="batch", fil=rng.randint(16, 256), per=rng.randint(200, 400), per_hi=rng.randint(500, 900))
        return _case(call="batch", fil=rng.randint(8, 64), per=1000, per_hi=int(_log(rng, 4000, 100000)))
    precision = "fp64" if call == "velocity fp64" or (call == "energy" and rng.random() < 0.4) else "mixed"
    top = {"velocity": 3e6, "host": 2e6, "rk4": 6e5, "energy": 8e5}.get(call, 6e4)
    if precision == "fp64":
        top = min(top, 6e4)
    N = _log(rng, 2e3, top)
    per = rng.randint(40, 260)
    fil = max(2, round(N / per))
    # modes per axis from 2.8 to 5.5 times N^(1/3), odd counts among them
    M = int(min(512, max(32, rng.uniform(2.8, 5.5) * (fil * per) ** (1 / 3))))
    if precision == "fp64":
        M = min(M, 160)
    box = rng.choice([1.0, 1.0, 1.25]) if M <= 420 else 1.0
    return _case(call="velocity" if call == "velocity fp64" else call, precision=precision, fil=fil, per=per, M=M,
                 ragged=rng.random() < 0.5, Q=rng.choice([2, 2, 3]), w=rng.choice([8, 8, 8, 6, 10]),
                 sigma=rng.choice([1.5, 1.5, 1.5, 2.0]) if M <= 256 else 1.5, box=box,
                 deterministic=call == "velocity" and rng.random() < 0.1)


# ------------------------------------------------------------------ inputs
def _box(c):
    return np.array([SIDE, SIDE * c["box"], SIDE])


def _sizes(c):
    """Node counts belong to the case, not to the seed: every seed gives outputs of one shape."""
    return np.random.default_rng([c["fil"], c["per"], c["per_hi"]])


def _tangle(gen, counts, L):
    """Random-phase Fourier curves, counts[f] nodes on curve f (as workloads.fourier_tangle, seeded on the GPU)."""
    dev, nfil, modes = "cuda", len(counts), 8
    n = torch.as_tensor(counts, device=dev)
    f = torch.repeat_interleave(torch.arange(nfil, device=dev), n)
    first = torch.cumsum(n, 0) - n
    th = 2 * math.pi * (torch.arange(f.numel(), device=dev) - first[f]).double() / n[f]
    kw = dict(generator=gen, device=dev, dtype=torch.float64)
    X = (torch.rand((nfil, 3), **kw) * torch.as_tensor(L, device=dev))[f]
    for m in range(1, modes + 1):
        u, v = (torch.randn((2, nfil, 3), **kw) * (float(L.min()) / 128 / m)).unbind(0)
        X += u[f] * torch.cos(m * th)[:, None] + v[f] * torch.sin(m * th)[:, None]
    return X


def _curves(c, seed):
    """Node positions (on the GPU) and filament offsets of a single configuration."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    rng = np.random.default_rng(seed)
    L, per, fil = _box(c), c["per"], c["fil"]
    counts = _sizes(c).integers(per // 2, 3 * per // 2 + 1, fil) if c["ragged"] else np.full(fil, per)
    offsets = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    if c["shape"] == "tangle":
        return _tangle(gen, counts, L), offsets
    th = 2 * math.pi * (np.arange(per) + rng.uniform()) / per
    ring = np.stack([np.cos(th), np.sin(th), 0 * th], 1)
    curves = []
    for k in range(fil):
        center = rng.uniform(0, 1, 3) * L
        if c["shape"] == "leapfrog":  # coaxial ellipses normal to x, a quarter of the box apart
            a, b = (SIDE / 4 * math.sqrt(2), SIDE / 4) if k == 0 else (SIDE / 4, SIDE / 4 * math.sqrt(2))
            if k == 0:
                at = center
            X = at + np.array([k * SIDE / 4, 0, 0]) + np.stack([ring[:, 2], a * ring[:, 0], b * ring[:, 1]], 1)
        elif c["shape"] == "ring":
            X = center + SIDE / 6 * ring
        else:
            frame = np.linalg.qr(rng.standard_normal((3, 3)))[0]
            X = center + (ring * np.array([*rng.uniform(0.5, 1.5, 2), 0])) @ frame.T
        curves.append(X)
    return torch.from_numpy(np.concatenate(curves)).cuda(), offsets


def _batch(c, seed):
    """The members' nodes and offsets."""
    rng, sizes = np.random.default_rng(seed), _sizes(c)
    got = []
    for k in range(c["fil"]):
        n = int(round(math.exp(sizes.uniform(math.log(c["per"]), math.log(c["per_hi"])))))
        nfil = max(2, round(n / 100)) if c["per"] >= 1000 else int(sizes.integers(3, 8))
        per = n // nfil
        gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 62)))
        got.append((_tangle(gen, np.full(nfil, per), _box(c)), np.arange(nfil + 1, dtype=np.int64) * per))
    return got


def _params(c):
    L = _box(c)
    flags = (B.BS_WANT_PSI if c["call"] == "energy" else 0) | (B.BS_DETERMINISTIC if c["deterministic"] else 0)
    p = B.make_params(L, kappa=KAPPA, a=CORE, delta=DELTA, beta=BETA, M=c["M"], Q=c["Q"], order=c["order"], w=c["w"],
                      sigma=c["sigma"], local_frac=c["local_frac"], flags=flags,
                      precision=B.BS_FP64 if c["precision"] == "fp64" else B.BS_MIXED)
    for d in range(3):  # the same k_max along a longer side
        p.M[d] = c["M"] if L[d] == L.min() else int(math.ceil(c["M"] * L[d] / L.min())) | 1
    return p


def _time_step(nodes, offsets):
    """The Kelvin-wave step at the smallest node spacing."""
    x = nodes.cpu().numpy()
    after = np.arange(1, len(x) + 1)
    after[offsets[1:] - 1] = offsets[:-1]
    return B.kelvin_wave_period(np.linalg.norm(x[after] - x, axis=1).min(), KAPPA, CORE, DELTA)


def prepare(case, seed):
    c = dict(_PLAIN, **case)
    s = {"call": c["call"]}
    if c["call"] == "batch":
        members = _batch(c, seed)
        params = [B.tangle_params(len(x), _box(c), beta=BETA, M_min=32, M_max=128, Q=c["Q"], w=c["w"], sigma=c["sigma"],
                                  precision=B.BS_MIXED) for x, _ in members]

        class Member:
            def __init__(self, offsets):
                self.offsets, self.closing = offsets, None

        s["stream"] = torch.cuda.Stream()
        s["bs"] = B.BiotSavartBatch(params, [Member(o) for _, o in members], stream=s["stream"])
        s["nodes"] = torch.cat([x for x, _ in members])
        s["vel"] = torch.empty_like(s["nodes"])
        torch.cuda.synchronize()
        return s
    nodes, offsets = _curves(c, seed)
    if c["call"] == "rk4":
        s["stream"] = torch.cuda.Stream()
        s["bs"] = B.BiotSavart(_params(c), offsets, stream=s["stream"])
        s["start"], s["nodes"] = nodes, nodes.clone()
        torch.cuda.synchronize()
        s["bs"].rk4_capture(s["nodes"], _time_step(nodes, offsets))
        return s
    s["bs"] = B.BiotSavart(_params(c), offsets)
    s["nodes"] = nodes
    if c["call"] == "host":
        s["nodes"] = nodes.cpu().pin_memory()
        s["vel"] = torch.empty_like(s["nodes"]).pin_memory()
    elif c["call"] == "energy":
        s["vel"], s["psi"] = torch.empty_like(nodes), torch.empty_like(nodes)
    return s


def run(s):
    if s["call"] == "velocity":
        return s["bs"].velocity(s["nodes"])
    if s["call"] == "energy":
        return {"energy": s["bs"].energy(s["nodes"], s["vel"], s["psi"]), "vel": s["vel"], "psi": s["psi"]}
    if s["call"] == "host":
        B.bs_compute_host(s["bs"].ctx, s["nodes"], s["vel"])
        return s["vel"]
    with torch.cuda.stream(s["stream"]):
        if s["call"] == "batch":
            out = s["bs"].velocity(s["nodes"], s["vel"])
        else:
            out = s["nodes"].copy_(s["start"])  # every pass steps from the same positions
            s["bs"].rk4_launch(1)
    torch.cuda.current_stream().wait_stream(s["stream"])
    return out


def work(case):
    """Nodes read and velocities written once, in float64; the pair terms inside the cut-off at uniform density (30
    operations each), the transforms of three components both ways (5 n log2 n, half for real data) on the mode grid
    times sigma, the spread and the interpolation (6 w^3 a point), for each evaluation."""
    c = dict(_PLAIN, **case)

    def one(N, M, n_eval, extra):
        rc = BETA * 2 * BETA / max(1, (M - 1) // 2) * SIDE / (2 * math.pi)
        pairs = N * c["Q"] * N * min(1.0, 4 * math.pi / 3 * rc ** 3 / (SIDE ** 3 * c["box"]))
        n3 = (c["sigma"] * M) ** 3 * c["box"]
        fft = 2 * 3 * 2.5 * n3 * math.log2(n3)
        return np.array([48.0 * N + extra * N, n_eval * (30 * pairs + fft + 6 * c["w"] ** 3 * N * (c["Q"] + 1))])

    if c["call"] == "batch":
        mid = math.sqrt(c["per"] * c["per_hi"])
        N = (c["per_hi"] - c["per"]) / math.log(c["per_hi"] / c["per"])
        both = c["fil"] * one(N, min(128, max(32, 2.8 * mid ** (1 / 3))), 1, 0)
    else:
        both = one(c["fil"] * c["per"], c["M"], 4 if c["call"] == "rk4" else 1, 24 if c["call"] == "energy" else 0)
    return {"bytes": float(both[0]), "flops": float(both[1])}


# ------------------------------------------------- the same sums in 64 bits
def _splines(x, offsets, order):
    """Coefficients (N, order, 3) in the local chord-length parameter and chord lengths of the periodic splines
    through the nodes: end derivatives from the continuity of the next two (cubic: one) derivatives."""
    N = len(x)
    C, H = np.zeros((N, order, 3)), np.zeros(N)
    for a, b in zip(offsets[:-1], offsets[1:]):
        p, n = x[a:b], b - a
        D = np.roll(p, -1, axis=0) - p
        h = np.linalg.norm(D, axis=1)
        i, nx = np.arange(n), np.roll(np.arange(n), -1)
        H[a:b] = h
        hc = h[:, None]
        if order == 4:  # end derivatives d: second derivative at the start and the end of each segment
            A, R = np.zeros((n, n)), np.zeros((n, 3))
            np.add.at(A, (nx, i), 2 / h)            # end of segment i, at node i + 1
            np.add.at(A, (nx, nx), 4 / h)
            np.add.at(A, (i, i), 4 / h)             # minus the start of segment i, at node i
            np.add.at(A, (i, nx), 2 / h)
            R += 6 * D / hc ** 2
            np.add.at(R, nx, 6 * D / hc ** 2)
            d0 = np.linalg.solve(A, R)
            d1 = d0[nx]
            C[a:b] = np.stack([p, d0, (3 * D / hc - 2 * d0 - d1) / hc, (d0 + d1 - 2 * D / hc) / hc ** 2], 1)
            continue
        # quintic: end first and second derivatives d, e; third and fourth derivatives continuous
        A, R = np.zeros((2 * n, 2 * n)), np.zeros((2 * n, 3))
        for row, col, v in ((nx, i, -24 / h ** 2), (nx, nx, -36 / h ** 2), (nx, n + i, -3 / h), (nx, n + nx, 9 / h),
                            (i, i, 36 / h ** 2), (i, nx, 24 / h ** 2), (i, n + i, 9 / h), (i, n + nx, -3 / h),
                            (n + nx, i, -168 / h ** 3), (n + nx, nx, -192 / h ** 3), (n + nx, n + i, -24 / h ** 2),
                            (n + nx, n + nx, 36 / h ** 2), (n + i, i, -192 / h ** 3), (n + i, nx, -168 / h ** 3),
                            (n + i, n + i, -36 / h ** 2), (n + i, n + nx, 24 / h ** 2)):
            np.add.at(A, (row, col), v)
        np.add.at(R, nx, -60 * D / hc ** 3)
        np.add.at(R, i, 60 * D / hc ** 3)
        np.add.at(R, n + nx, -360 * D / hc ** 4)
        np.add.at(R, n + i, -360 * D / hc ** 4)
        scale = np.concatenate([np.ones(n), np.full(n, 1 / h.mean())])[:, None]  # unknowns and rows of like size
        S = scale * np.linalg.solve(A * scale.T / scale, R / scale)
        d0, e0 = S[:n], S[n:]
        d1, e1 = d0[nx], e0[nx]
        C[a:b] = np.stack([p, d0, e0 / 2, (20 * D - (8 * d1 + 12 * d0) * hc - (3 * e0 - e1) * hc ** 2) / (2 * hc ** 3),
                           (-30 * D + (14 * d1 + 16 * d0) * hc + (3 * e0 - 2 * e1) * hc ** 2) / (2 * hc ** 4),
                           (12 * D - 6 * (d1 + d0) * hc + (e1 - e0) * hc ** 2) / (2 * hc ** 5)], 1)
    return C, H


def _points(C, H, u):
    """Positions and tau-derivatives at the fractions u of every segment: (N, len(u), 3) each."""
    t = H[:, None] * u[None, :]
    k = np.arange(C.shape[1])
    X = np.einsum("nqk,nkc->nqc", t[:, :, None] ** k, C)
    V = np.einsum("nqk,nkc->nqc", k[1:] * t[:, :, None] ** (k[1:] - 1), C[:, 1:])
    return X, V


def _sums(x, offsets, L, Q, order, frac):
    """Velocity and streamfunction at the nodes x: the quadrature-discretised periodic sums, converged (Ewald's split
    at beta = 6, so that what it leaves out is below 1e-15)."""
    C, H = _splines(x, offsets, order)
    N = len(x)
    g, gw = np.polynomial.legendre.leggauss(Q)
    g, gw = (g + 1) / 2, gw / 2
    before = np.arange(N) - 1
    before[offsets[:-1]] = offsets[1:] - 1
    X, V = _points(C, H, g)
    q = V * (gw[None, :, None] * H[:, None, None])
    # local terms: Taylor expansion on the fraction f next to the node, plain quadrature on the rest
    f = frac or 1.0
    lp = f * H * (np.linalg.norm(_points(C, H, f * g)[1], axis=2) @ gw)
    lm = (f * H * (np.linalg.norm(_points(C, H, 1 - f * g)[1], axis=2) @ gw))[before]
    d, dd = C[:, 1], 2 * C[:, 2]
    sn = np.linalg.norm(d, axis=1)[:, None]
    lg = np.log(2 * np.sqrt(lm * lp) / CORE)[:, None]
    vel = KAPPA / (4 * math.pi) * np.cross(d, dd) / sn ** 3 * (lg - DELTA)
    psi = KAPPA / (2 * math.pi) * d / sn * (lg - (DELTA - 1))
    pre = KAPPA / (4 * math.pi)
    lo = f
    while lo < 1:
        hi = min(1.0, 2 * lo)
        hi = 1.0 if 1 - hi < 1e-12 else hi
        u = lo + (hi - lo) * g
        for seg, uu in ((np.arange(N), u), (before, 1 - u)):
            Y, W = _points(C[seg], H[seg], uu)
            r = Y - x[:, None]
            W = W * (gw * (hi - lo))[None, :, None] * H[seg][:, None, None]
            rn = np.linalg.norm(r, axis=2)[:, :, None]
            vel += pre * (np.cross(r, W) / rn ** 3).sum(1)
            psi += pre * (W / rn).sum(1)
        lo = hi
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    t64 = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
    alpha = 6.0 / float(L.min())
    src, chg, tgt, Lt = t64(X.reshape(-1, 3)), t64(q.reshape(-1, 3)), t64(x), t64(L)
    vel, psi = t64(vel), t64(psi)
    own = torch.as_tensor(np.stack([np.arange(N), before], 1), device=dev)
    images = torch.cartesian_prod(*[torch.arange(-1.0, 2.0, device=dev, dtype=torch.float64)] * 3) * Lt
    step = max(1, int(2e7 / len(src)))
    seg = torch.arange(N, device=dev).repeat_interleave(Q)
    c2 = 2 * alpha / math.sqrt(math.pi)
    for a in range(0, N, step):
        b = min(N, a + step)
        D = src[None] - tgt[a:b, None]
        D = D - Lt * torch.round(D / Lt)
        local = (seg[None] == own[a:b, :1]) | (seg[None] == own[a:b, 1:])
        for im in images:
            R = D + im
            r = R.square().sum(2).sqrt()
            ga = c2 * r * torch.exp(-(alpha * r) ** 2)
            short, by_r = torch.erfc(alpha * r), 1 / r
            gv, gp = (short + ga) * by_r ** 3, short * by_r
            if not im.any():  # C_0: the long-range field's share is taken off in its place
                gv = torch.where(local, (ga - torch.erf(alpha * r)) * by_r ** 3, gv)
                gp = torch.where(local, -torch.erf(alpha * r) * by_r, gp)
            S = torch.einsum("tsi,sj,ts->tij", R, chg, gv)
            vel[a:b] += pre * torch.stack([S[:, 1, 2] - S[:, 2, 1], S[:, 2, 0] - S[:, 0, 2], S[:, 0, 1] - S[:, 1, 0]], 1)
            psi[a:b] += pre * gp @ chg
    # long range: direct sums over the modes that matter
    K = [int(math.ceil(6 * alpha * l / math.pi)) for l in L]
    k = [torch.arange(-K[i], K[i] + 1, device=dev, dtype=torch.float64) * (2 * math.pi / L[i]) for i in range(3)]
    phase = lambda y: [torch.polar(torch.ones((), device=dev, dtype=torch.float64), y[:, i:i + 1] * k[i]) for i in range(3)]  # noqa: E731
    kx, ky, kz = torch.meshgrid(*k, indexing="ij")
    k2 = kx ** 2 + ky ** 2 + kz ** 2
    k2[K[0], K[1], K[2]] = 1
    gauss = torch.exp(-k2 / (4 * alpha ** 2)) / k2
    gauss[K[0], K[1], K[2]] = 0
    om = torch.zeros((3, *k2.shape), dtype=torch.complex128, device=dev)
    step = 4000
    for a in range(0, len(src), step):
        e = [p.conj() for p in phase(src[a:a + step])]
        xy = (e[0][:, :, None] * e[1][:, None, :]).reshape(len(e[0]), -1)
        for i in range(3):
            om[i] += (xy.T @ (e[2] * chg[a:a + step, i:i + 1])).reshape(k2.shape)
    om *= KAPPA / float(np.prod(L)) * gauss
    vk = 1j * torch.stack([ky * om[2] - kz * om[1], kz * om[0] - kx * om[2], kx * om[1] - ky * om[0]])
    for a in range(0, N, step):
        e = phase(tgt[a:a + step])
        xy = (e[0][:, :, None] * e[1][:, None, :]).reshape(len(e[0]), -1)
        for i in range(3):
            vel[a:a + step, i] += ((xy @ vk[i].reshape(xy.shape[1], -1)) * e[2]).sum(1).real
            psi[a:a + step, i] += ((xy @ om[i].reshape(xy.shape[1], -1)) * e[2]).sum(1).real
    return vel, psi


def exact(case, seed):
    c = dict(_PLAIN, **case)
    if c["call"] == "batch":
        if c["fil"] * c["per_hi"] > 300000:
            return None
        return torch.cat([_sums(x.cpu().numpy(), o, _box(c), c["Q"], 4, 0.0)[0] for x, o in _batch(c, seed)])
    if c["fil"] * c["per"] > 12000 or (c["call"] == "rk4" and c["fil"] * c["per"] > 5000):
        return None
    nodes, offsets = _curves(c, seed)
    x = nodes.cpu().numpy()

    def at(y):
        return _sums(y, offsets, _box(c), c["Q"], c["order"], c["local_frac"])

    if c["call"] == "rk4":
        dt, k = _time_step(nodes, offsets), []
        for h in (0, dt / 2, dt / 2, dt):
            k.append(at(x + h * k[-1] if k else x)[0].cpu().numpy())
        return torch.from_numpy(x + dt / 6 * (k[0] + 2 * (k[1] + k[2]) + k[3]))
    vel, psi = at(x)
    # the energy's line integral interpolates the streamfunction in a way of its own: no value for it
    return {"energy": None, "vel": vel, "psi": psi} if c["call"] == "energy" else vel
