"""GPU parity of the 2D tile kernel (several steps per launch in shared memory)
against the oracle: lattices smaller than a tile, ragged and odd ones, one CTA
and many, both tile shapes, step counts that leave every remainder, every coin
class, phase coins, the three shifts, edges, fixed and random links, walkers
whose window wraps or meets the edges.  Tolerance: amp_tol."""
import numpy as np
import pytest

import oracle
from paper_1003_3779_gb300 import inputs
from tests.helpers import amp_tol, maxabs

pytestmark = pytest.mark.gpu

DIMS = [(1, 1), (2, 3), (1, 40), (33, 1), (17, 31), (32, 32), (65, 33), (129, 50)]


@pytest.fixture(scope="module")
def qw():
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    return qw


def coin_named(name):
    rng = np.random.default_rng(len(name))
    if name == "real":
        q, _ = np.linalg.qr(rng.standard_normal((4, 4)))
        return q.astype(np.complex128)
    return {"grover": inputs.grover(), "hh": inputs.hadamard2(), "complex": inputs.random_unitary(4, rng)}[name]


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("coin", ["grover", "hh", "real", "complex"])
@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("phases", [False, True])
def test_periodic(qw, dims, coin, shift, phases):
    Lx, Ly = dims
    C = coin_named(coin)
    psi0 = inputs.random_state((4, Ly, Lx), seed=51)
    phi = np.random.default_rng(52).uniform(-3, 3, size=(Lx * Ly, 4)).astype(np.float32) if phases else None
    for k, T in ((8, 1), (8, 7), (8, 21), (4, 6)):
        want = oracle.evolve(psi0, C, T, shift=shift, phi=None if phi is None else phi.astype(np.float64))
        w = qw.Walk(dims, prec="f32", shift=shift)
        w.set_coin(C) if phi is None else w.set_coin_phases(C, phi)
        w.set_plan(k).set_state(psi0)
        assert maxabs(w.step(T).state(), want) < amp_tol("f32", T)
        w.close()


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("bc", [0, 1, 2])
@pytest.mark.parametrize("noise,fixed", [(0.0, 0.0), (0.0, 0.3), (0.2, 0.0), (0.1, 0.1), (1.0, 0.0)])
def test_links_and_edges(qw, dims, shift, bc, noise, fixed):
    Lx, Ly = dims
    ns, T, seed, t0 = Lx * Ly, 15, 0x9ABC_DEF0_1234_5678, 3
    rng = np.random.default_rng(53)
    psi0 = inputs.random_state((4, Ly, Lx), seed=54)
    mask = (rng.uniform(size=(2, ns)) < fixed).astype(np.uint8)
    closed = np.broadcast_to(mask, (T, 2, ns)).copy()
    if noise:
        closed |= oracle.link_masks((Ly, Lx), seed, noise, t0, T)
    for coin, phases in (("grover", False), ("complex", False), ("complex", True)):
        C = coin_named(coin)
        phi = rng.uniform(-3, 3, size=(ns, 4)).astype(np.float32) if phases else None
        want = oracle.evolve(psi0, C, T, shift=shift, bc=bc, closed=closed, closed_per_step=True,
                             phi=None if phi is None else phi.astype(np.float64))
        w = qw.Walk(dims, prec="f32", shift=shift, bc=bc)
        w.set_coin(C) if phi is None else w.set_coin_phases(C, phi)
        if fixed:
            w.set_links(mask)
        w.set_link_noise(noise, seed, t0).set_state(psi0)
        assert maxabs(w.step(T).state(), want) < amp_tol("f32", T)
        w.close()


@pytest.mark.parametrize("bc,noise", [(0, 0.0), (0, 0.1), (1, 0.1), (2, 0.0)])
def test_large_tiles(qw, bc, noise):
    """Boxes of many tiles take the 64 x 64 shape: dense, and a window near a corner."""
    Lx, Ly, T, seed = 1500, 900, 13, 5
    C = inputs.grover()
    closed = oracle.link_masks((Ly, Lx), seed, noise, 0, T) if noise else None
    phi = inputs.region_grad_phases(1500, seed=6)[:Ly].reshape(-1, 4).astype(np.float32)
    for psi0 in (inputs.random_state((4, Ly, Lx), seed=55), inputs.localized_2d(Lx, 3, Ly - 2, Ly=Ly)):
        want = oracle.evolve(psi0, C, T, bc=bc, closed=closed, closed_per_step=closed is not None, phi=phi.astype(np.float64))
        w = qw.Walk((Lx, Ly), prec="f32", bc=bc).set_coin_phases(C, phi).set_link_noise(noise, seed).set_state(psi0)
        assert maxabs(w.step(T).state(), want) < amp_tol("f32", T)
        w.close()
