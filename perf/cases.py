"""The work that users of the walk library have it do, as cases to be timed.

Each case is one call sequence of a user's program: hand over a state (or the
coins and starting sites, or the phases), advance the walk, read the outputs
back into device tensors.  Sizes and distributions are those of the library's
workloads (``paper_1003_3779_gb300/inputs.py``): the 2001-site Hadamard cycle,
the 2^27-site SU(2) cycle, the 8192^2 torus, the batch of 4096 walks, the
1024^2 gradient and the random 4-regular graph, with smaller and odd sizes of
the same kinds beside them.

A case is a dict of plain values with a ``kind``:

* ``site1d``   a walker on one site of a cycle, a segment or a line
* ``cycle``    a random state on the cycle, one coin for all sites, autotuned
* ``torus``    a random state on the torus, one coin for all sites, autotuned
* ``site2d``   a walker on one site of the torus
* ``links``    a torus or a cut-out of the plane whose links break at random
* ``grad``     the gradient of a region's probability with respect to phases
* ``batch``    many independent localised walks in one launch, autotuned
* ``graph``    a random 4-regular graph, Grover coin, autotuned
"""
import math

import numpy as np
import torch

from paper_1003_3779_gb300 import qw

DEV = "cuda"
BC = {"periodic": 0, "segment": 1, "line": 2}
SHIFT = {"moving": 0, "flipflop": 1, "diagonal": 2}
REAL = {"f32": torch.float32, "f64": torch.float64, "comp": torch.float64}
CPLX = {"f32": torch.complex64, "f64": torch.complex128, "comp": torch.complex128}
LINK_P, LINK_SEED = 0.05, 7


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the small Hadamard cycle in double precision: a call of a millisecond,
        # where launches and latency count
        {"name": "cycle_site_2001_f64", "kind": "site1d", "n": 2001, "t": 1000, "prec": "f64", "bc": "periodic"},
        # the paper's line computation: a walker in the middle of a line that
        # absorbs at its ends
        {"name": "line_site_1m_f32", "kind": "site1d", "n": 1 << 20, "t": 1024, "prec": "f32", "bc": "line"},
        # the largest cycle: the workload the throughput metric is quoted on
        {"name": "cycle_2p27_f32", "kind": "cycle", "n": 1 << 27, "t": 4096, "prec": "f32", "theta": math.pi / 4,
         "xi": 0.0, "zeta": 0.0, "shift": "moving", "adjoint": False},
        # an ordinary cycle of odd length with a complex coin
        {"name": "cycle_1000003_complex_f32", "kind": "cycle", "n": 1000003, "t": 1000, "prec": "f32",
         "theta": 0.7853, "xi": 0.3, "zeta": -0.2, "shift": "moving", "adjoint": False},
        # the double-precision form on an ordinary cycle, run backward
        {"name": "cycle_1m_adjoint_f64", "kind": "cycle", "n": 1 << 20, "t": 1024, "prec": "f64", "theta": 0.3,
         "xi": 0.0, "zeta": 0.0, "shift": "moving", "adjoint": True},
        # the large torus with the Grover coin
        {"name": "torus_8192_grover_f32", "kind": "torus", "nx": 8192, "ny": 8192, "t": 1024, "prec": "f32",
         "coin": "grover", "shift": "moving"},
        # a small torus, not square, sides no power of two
        {"name": "torus_300x200_grover_f32", "kind": "torus", "nx": 300, "ny": 200, "t": 200, "prec": "f32",
         "coin": "grover", "shift": "flipflop"},
        # the paper's 2D timings: a walker on one site of the diagonal lattice
        {"name": "torus_site_diagonal_f32", "kind": "site2d", "nx": 8192, "ny": 8192, "t": 500, "prec": "f32",
         "coin": "hadamard2", "shift": "diagonal"},
        # links that break at random at every step, reflecting ends
        {"name": "links_2048x1500_f32", "kind": "links", "nx": 2048, "ny": 1500, "t": 64, "prec": "f32",
         "bc": "segment", "shift": "moving"},
        # the gradient with respect to every site's phases
        {"name": "grad_1024_f32", "kind": "grad", "l": 1024, "t": 512, "k": 64, "prec": "f32"},
        # thousands of walks of uneven length in one launch
        {"name": "batch_4096_f32", "kind": "batch", "walks": 4096, "nmax": 65536, "tmax": 4096, "sizes": 3},
        # a random 4-regular graph: no locality
        {"name": "graph_4m_f32", "kind": "graph", "vertices": 1 << 22, "t": 20, "prec": "f32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["site1d", "cycle", "cycle", "torus", "torus", "site2d", "links", "grad", "batch", "graph"])
    if kind == "site1d":
        return {"kind": kind, "n": _log(rng, 101, 1 << 20), "t": _log(rng, 64, 2048), "prec": rng.choice(["f64", "f32"]),
                "bc": rng.choice(["periodic", "segment", "line"])}
    if kind == "cycle":
        prec = rng.choice(["f32", "f32", "f64", "comp"])
        t = _log(rng, 64, 4096)
        top = (1 << 27) if prec == "f32" else (1 << 32) // t    # the wider forms are far slower
        n = _log(rng, 20000, min(1 << 26, top))
        cplx = rng.random() < 0.5
        return {"kind": kind, "n": n, "t": t, "prec": prec, "theta": round(rng.uniform(0.1, 1.4), 4),
                "xi": round(rng.uniform(-1, 1), 3) if cplx else 0.0, "zeta": round(rng.uniform(-1, 1), 3) if cplx else 0.0,
                "shift": rng.choice(["moving", "flipflop"]), "adjoint": rng.random() < 0.3}
    if kind == "torus":
        return {"kind": kind, "nx": _log(rng, 64, 8192), "ny": _log(rng, 64, 8192), "t": _log(rng, 16, 1024),
                "prec": "f32", "coin": rng.choice(["grover", "hadamard2"]),
                "shift": rng.choice(["moving", "flipflop", "diagonal"])}
    if kind == "site2d":
        return {"kind": kind, "nx": _log(rng, 256, 8192), "ny": _log(rng, 256, 8192), "t": _log(rng, 32, 500),
                "prec": "f32", "coin": rng.choice(["grover", "hadamard2"]),
                "shift": rng.choice(["moving", "flipflop", "diagonal"])}
    if kind == "links":
        return {"kind": kind, "nx": _log(rng, 64, 4096), "ny": _log(rng, 64, 4096), "t": _log(rng, 16, 128),
                "prec": "f32", "bc": rng.choice(["periodic", "segment", "line"]),
                "shift": rng.choice(["moving", "flipflop"])}
    if kind == "grad":
        return {"kind": kind, "l": _log(rng, 100, 1024), "t": _log(rng, 64, 512), "k": rng.choice([32, 64]),
                "prec": "f32"}
    if kind == "batch":
        return {"kind": kind, "walks": _log(rng, 64, 4096), "nmax": _log(rng, 1024, 65536), "tmax": _log(rng, 256, 4096),
                "sizes": rng.randrange(1 << 20)}
    return {"kind": kind, "vertices": _log(rng, 1 << 13, 1 << 22), "t": _log(rng, 4, 50),
            "prec": rng.choice(["f32", "f32", "f64"])}


# ---------------------------------------------------------------- inputs
def _su2(theta, xi=0.0, zeta=0.0):
    c, s = math.cos(theta), math.sin(theta)
    return np.array([[np.exp(1j * xi) * c, np.exp(1j * zeta) * s], [-np.exp(-1j * zeta) * s, np.exp(-1j * xi) * c]])


def _coin(case):
    if case["kind"] == "cycle":
        return _su2(case["theta"], case["xi"], case["zeta"])
    h = np.array([[1, 1], [1, -1]], complex) / math.sqrt(2.0)
    if case["kind"] == "site1d":
        return h
    return np.kron(h, h) if case.get("coin") == "hadamard2" else np.full((4, 4), 0.5, complex) - np.eye(4)


def _shape(case):
    if case["kind"] in ("site1d", "cycle"):
        return (2, case["n"])
    if case["kind"] == "grad":
        return (4, case["l"], case["l"])
    if case["kind"] == "graph":
        return (4 * case["vertices"],)
    return (4, case["ny"], case["nx"])


def _rng(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _random_state(shape, seed, dtype):
    """i.i.d. complex Gaussian amplitudes over their norm, on the device."""
    z = torch.randn(shape, generator=_rng(seed), device=DEV, dtype=dtype)
    n2 = sum(float(p.abs().double().square().sum()) for p in (z if z.dim() > 1 else z[None]))
    return z.mul_(1.0 / math.sqrt(n2))


def _site(case, seed):
    """(column, row) of the walker: within a tenth of the middle, by the seed."""
    r = np.random.RandomState(seed % (1 << 31))
    nx, ny = case.get("nx", case.get("n")), case.get("ny", 1)
    return (nx // 2 + int(r.randint(-(nx // 10), nx // 10 + 1)), ny // 2 + int(r.randint(-(ny // 10), ny // 10 + 1)))


def _coin_state(d, seed):
    """A random normalised coin state, by the seed."""
    r = np.random.RandomState((seed + 1) % (1 << 31))
    v = r.standard_normal(d) + 1j * r.standard_normal(d)
    return v / np.linalg.norm(v)


def _state(case, seed):
    """The state that the program hands over: a device tensor of d planes."""
    dtype, shape = CPLX[case["prec"]], _shape(case)
    if case["kind"] in ("site1d", "site2d"):
        psi = torch.zeros(shape, dtype=dtype, device=DEV)
        x, y = _site(case, seed)
        v = torch.from_numpy(_coin_state(shape[0], seed)).to(DEV, dtype)
        if case["kind"] == "site1d":
            psi[:, x] = v
        else:
            psi[:, y, x] = v
        return psi
    if case["kind"] == "grad":   # the workload's start: one site in the lattice's corner
        psi = torch.zeros(shape, dtype=dtype, device=DEV)
        psi[:, 0, 0] = torch.tensor([0.5, -0.5, -0.5, 0.5], dtype=dtype, device=DEV)
        return psi
    return _random_state(shape, seed, dtype)


def _phases(case, seed):
    l = case["l"]
    return (torch.rand((l * l, 4), generator=_rng(seed), device=DEV) - 0.5) * 0.2


def _rect(case):
    l = case["l"]
    s = max(4, l // 16)
    return (l // 4 - s // 2, l // 4 - s // 2, s, s)


def _batch_params(case, seed):
    """Sizes and lengths belong to the case; coins and starting sites to the seed."""
    r = np.random.RandomState(case["sizes"])
    n = r.randint(min(256, case["nmax"]), case["nmax"] + 1, case["walks"]).astype(np.int64)
    t = r.randint(min(64, case["tmax"]), case["tmax"] + 1, case["walks"]).astype(np.int64)
    r = np.random.RandomState(seed % (1 << 31))
    theta = r.uniform(0.0, math.pi / 2, case["walks"])
    x0 = np.minimum((r.uniform(0.0, 1.0, case["walks"]) * n).astype(np.int64), n - 1)
    return n, t, theta, x0


def _matching(case, seed):
    """partner of each arc: a random perfect matching of the vertices' edge ends."""
    a = 4 * case["vertices"]
    perm = torch.randperm(a, generator=_rng(seed), device=DEV)
    partner = torch.empty(a, dtype=torch.int64, device=DEV)
    partner[perm[0::2]] = perm[1::2]
    partner[perm[1::2]] = perm[0::2]
    return partner


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        n, t, theta, x0 = _batch_params(case, seed)
        b = qw.Batch(n, t, np.stack([_su2(th) for th in theta]), x0)
        b.autotune()
        return {"case": case, "b": b, "P": torch.empty(int(n.sum()), dtype=torch.float32, device=DEV)}
    psi = _state(case, seed)
    out = torch.empty_like(psi)
    if kind == "graph":
        off = np.arange(0, 4 * case["vertices"] + 1, 4, dtype=np.int64)
        g = qw.GraphWalk(off, _matching(case, seed).cpu().numpy(), prec=case["prec"])
        g.set_state(psi)
        g.autotune()
        return {"case": case, "w": g, "psi": psi, "out": out}
    dims = tuple(reversed(psi.shape[1:]))
    w = qw.Walk(dims, prec=case["prec"], shift=SHIFT[case.get("shift", "moving")], bc=BC[case.get("bc", "periodic")])
    if kind == "grad":
        phi = _phases(case, seed).requires_grad_(True)
        return {"case": case, "w": w, "psi": psi, "phi": phi, "base": _coin(case)}
    w.set_coin(_coin(case))
    if kind == "links":
        w.set_link_noise(LINK_P, LINK_SEED)
    if kind in ("cycle", "torus"):
        w.set_state(psi)
        w.autotune()
    P = torch.empty(psi.shape[1:], dtype=REAL[case["prec"]], device=DEV)
    return {"case": case, "w": w, "psi": psi, "out": out, "P": P}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        P, norms = state["b"].step().probabilities(state["P"])
        return {"P": P, "norms": norms.astype(np.float32)}   # a norm is a sum of float probabilities
    w = state["w"]
    if case["kind"] == "grad":
        phi = state["phi"]
        phi.grad = None
        loss = qw.region_mass(phi, w, state["base"], state["psi"], _rect(case), case["t"], case["k"])
        loss.backward()
        return {"loss": loss.detach().float(), "grad": phi.grad}   # the walk is in float
    if case["kind"] == "links":
        w.set_link_noise(LINK_P, LINK_SEED)   # the same links again on every pass
    w.set_state(state["psi"])
    if case.get("adjoint"):
        w.step_adjoint(case["t"])
    else:
        w.step(case["t"])
    if case["kind"] == "graph":
        return {"psi": w.state(out=state["out"])}
    qw.qw_probabilities(w.h, state["P"], want_norm=False)
    return {"psi": qw.qw_get_state(w.h, state["out"]), "P": state["P"]}


# ---------------------------------------------------------------- what a pass cannot do without
def _cone(n, t, periodic=True):
    """Site-steps of the light cone of one site on a cycle of n sites."""
    tc = min(t, (n - 1) // 2)
    return tc * tc + (t - tc) * n


def work(case):
    kind, t = case["kind"], case["t"] if "t" in case else 0
    if kind == "batch":
        n, ts, _, _ = _batch_params(case, 0)
        return {"bytes": 4 * int(n.sum()) + 48 * len(n), "flops": 12 * sum(_cone(int(a), int(b)) for a, b in zip(n, ts))}
    amps = math.prod(_shape(case))
    sites = amps // (4 if kind == "graph" else _shape(case)[0])
    cb, rb = (8, 4) if case["prec"] == "f32" else (16, 8)
    if kind == "graph":   # amplitudes in and out, the partner of each arc; coin of each step
        return {"bytes": amps * (2 * cb + 4), "flops": 14 * amps // 2 * t}
    if kind == "grad":    # phases and state in, gradient out; forward, and two fields backward
        return {"bytes": 2 * 4 * 4 * sites + amps * cb, "flops": 3 * 28 * sites * t}
    io = amps * 2 * cb + sites * rb
    if kind in ("cycle", "torus"):   # one coin for all sites: transforms to momentum and back
        return {"bytes": io, "flops": int(2 * 5 * amps * math.log2(sites)) + 8 * _shape(case)[0] * amps}
    if kind == "site1d":
        return {"bytes": io, "flops": 8 * _cone(case["n"], t)}
    if kind == "site2d":
        cone = sum(min(2 * i + 1, case["nx"]) * min(2 * i + 1, case["ny"]) for i in range(t))
        return {"bytes": io, "flops": 28 * cone}
    return {"bytes": io, "flops": 28 * sites * t}


# ---------------------------------------------------------------- the same in 64 bits, by plain torch
def _momentum_power(coin, phases, conj, t, vec, flip):
    """vec <- (U^t or its adjoint) vec, U = S C at each momentum: row c of C times
    phases[c], stored in row c (c xor 1 for the flip-flop shift)."""
    d = len(phases)
    m = [[None] * d for _ in range(d)]
    for c in range(d):
        for k in range(d):
            m[c ^ 1 if flip else c][k] = phases[c] * complex(coin[c, k])
    if conj:
        m = [[m[k][c].conj() for k in range(d)] for c in range(d)]
    mul = lambda a, b: [[sum(a[i][k] * b[k][j] for k in range(d)) for j in range(d)] for i in range(d)]  # noqa: E731
    while t:
        if t & 1:
            vec = [sum(m[i][k] * vec[k] for k in range(d)) for i in range(d)]
        t >>= 1
        if t:
            m = mul(m, m)
    return vec


def _exact_lattice(case, psi):
    """One coin for all sites on a periodic lattice: in momentum space."""
    psi = psi.to(torch.complex128)
    flip, coin, t = case.get("shift") == "flipflop", _coin(case), case["t"]
    wave = lambda n: torch.exp(2j * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n)  # noqa: E731
    if psi.dim() == 2:
        f = [torch.fft.fft(p) for p in psi]
        ex = wave(psi.shape[1])
        f = _momentum_power(coin, [ex, ex.conj()], case.get("adjoint", False), t, f, flip)
        return torch.stack([torch.fft.ifft(p) for p in f])
    for p in psi:
        p.copy_(torch.fft.fft2(p))
    ny, nx = psi.shape[1:]
    ex, ey = wave(nx)[None, :], wave(ny)[:, None]
    rows = max(1, (1 << 21) // nx)
    for y in range(0, ny, rows):
        e = ey[y:y + rows]
        one = torch.ones_like(e) * torch.ones_like(ex)
        if case.get("shift") == "diagonal":
            ph = [ex.conj() * e.conj(), ex.conj() * e, ex * e.conj(), ex * e]
        else:
            ph = [ex.conj() * one, ex * one, e.conj() * one, e * one]
        f = _momentum_power(coin, ph, False, t, [psi[c, y:y + rows].clone() for c in range(4)], flip)
        for c in range(4):
            psi[c, y:y + rows] = f[c]
    for p in psi:
        p.copy_(torch.fft.ifft2(p))
    return psi


def _philox(sites, step):
    """Words 0 and 1 of Philox4x32-10 for counters (site, 0, step, 0) and key LINK_SEED."""
    m32 = 0xFFFFFFFF
    c0, c1 = sites & m32, sites >> 32
    c2, c3 = torch.full_like(sites, step), torch.zeros_like(sites)
    k0, k1 = LINK_SEED, 0
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((b >> 32) & m32) ^ c1 ^ k0, b & m32, ((a >> 32) & m32) ^ c3 ^ k1, a & m32
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c0, c1


def _exact_links(case, psi):
    """Links of a torus or a plane, closed at random; a closed link reflects, the ends
    of a line absorb."""
    psi = psi.to(torch.complex128)
    ny, nx = psi.shape[1:]
    coin = torch.from_numpy(_coin(case)).to(DEV)
    sites = torch.arange(nx * ny, device=DEV, dtype=torch.int64)
    thr = int(LINK_P * 4294967296.0)
    moving = case["shift"] == "moving"
    for t in range(case["t"]):
        wx, wy = (w.reshape(ny, nx) for w in _philox(sites, t))
        closed = [wx < thr, wy < thr]
        lost = [torch.zeros_like(closed[0]), torch.zeros_like(closed[1])]
        for axis, at in ((0, (slice(None), -1)), (1, (-1, slice(None)))):
            if case["bc"] == "segment":
                closed[axis][at] = True
            elif case["bc"] == "line":
                lost[axis][at] = True
                lost[axis] &= ~closed[axis]
        phi = torch.einsum("rc,cyx->ryx", coin, psi)
        out = []
        for c in range(4):
            axis, dim, sign = c >> 1, (1, 0)[c >> 1], 1 if c % 2 == 0 else -1
            # moving: the value arrives from v - e_c in coin c; flip-flop: from v + e_c in coin c xor 1
            s = -sign if moving else sign
            src, own = (c, c ^ 1) if moving else (c ^ 1, c)
            got = torch.roll(phi[src], -s, dim)
            shut, gone = (closed[axis], lost[axis]) if s > 0 else (torch.roll(closed[axis], 1, dim), torch.roll(lost[axis], 1, dim))
            out.append(torch.where(shut, phi[own], torch.where(gone, torch.zeros_like(got), got)))
        psi = torch.stack(out)
    return psi


def _exact_line(case, psi):
    psi = psi.to(torch.complex128)
    c = _coin(case)
    for _ in range(case["t"]):
        p0 = complex(c[0, 0]) * psi[0] + complex(c[0, 1]) * psi[1]
        p1 = complex(c[1, 0]) * psi[0] + complex(c[1, 1]) * psi[1]
        a, b = torch.roll(p0, -1), torch.roll(p1, 1)
        if case["bc"] == "segment":
            a[-1], b[0] = p1[-1], p0[0]
        elif case["bc"] == "line":
            a[-1], b[0] = 0, 0
        psi = torch.stack([a, b])
    return psi


def _exact_grad(case, seed):
    l, t = case["l"], case["t"]
    phase = torch.exp(1j * _phases(case, seed).double()).t().reshape(4, l, l).contiguous()
    coin = torch.from_numpy(_coin(case)).to(DEV)
    move = ((1, 1), (-1, 1), (1, 0), (-1, 0))
    psi, kept = _state(case, seed).to(torch.complex128), []
    for _ in range(t):
        kept.append(phase * psi)
        phi = torch.einsum("rc,cyx->ryx", coin, kept[-1])
        psi = torch.stack([torch.roll(phi[c], *move[c]) for c in range(4)])
    x, y, w, h = _rect(case)
    lam = torch.zeros_like(psi)
    lam[:, y:y + h, x:x + w] = psi[:, y:y + h, x:x + w]
    loss = lam.abs().square().sum()
    grad = torch.zeros((4, l, l), dtype=torch.float64, device=DEV)
    for b in reversed(kept):
        mu = torch.stack([torch.roll(lam[c], -move[c][0], move[c][1]) for c in range(4)])
        a = torch.einsum("rc,ryx->cyx", coin.conj(), mu)
        grad -= 2 * (a.conj() * b).imag
        lam = phase.conj() * a
    return {"loss": loss, "grad": grad.reshape(4, -1).t().contiguous()}


def _exact_batch(case, seed):
    ns, ts, thetas, x0s = _batch_params(case, seed)
    start = [complex(2 ** -0.5), 1j * 2 ** -0.5]
    got = []
    for n, t, th, x0 in zip(ns, ts, thetas, x0s):
        m = 1 << int(2 * t + 1).bit_length()     # a cycle that the cone does not go round
        ex = torch.exp(2j * math.pi * torch.arange(m, device=DEV, dtype=torch.float64) / m)
        one = torch.ones_like(ex)
        f = _momentum_power(_su2(th), [ex, ex.conj()], False, int(t), [s * one for s in start], False)
        psi = torch.fft.ifft(torch.stack(f))
        at = torch.arange(-int(t), int(t) + 1, device=DEV)
        full = torch.zeros((2, int(n)), dtype=torch.complex128, device=DEV)
        full.index_add_(1, (at + int(x0)) % int(n), psi[:, at % m])
        got.append(full.abs().square().sum(0))
    return {"P": torch.cat(got), "norms": torch.stack([p.sum() for p in got])}


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind == "grad":
        return _exact_grad(case, seed)
    psi = _state(case, seed)
    if kind == "graph":
        psi, partner = psi.to(torch.complex128), _matching(case, seed)
        for _ in range(case["t"]):
            v = psi.reshape(-1, 4)
            psi = (0.5 * v.sum(1, keepdim=True) - v).reshape(-1)[partner]
        return {"psi": psi}
    if kind == "links":
        psi = _exact_links(case, psi)
    elif kind == "site1d" and case["bc"] != "periodic":
        psi = _exact_line(case, psi)
    else:
        psi = _exact_lattice(case, psi)
    P = torch.zeros(psi.shape[1:], dtype=torch.float64, device=DEV)
    for p in psi:
        P += p.abs().square()
    return {"psi": psi, "P": P}
