"""GPU parity of the momentum-space steps of the cycle (qw_set_plan_ex variant 2)
against the FP64 oracle: blocks that wrap the cycle many times, ragged last
blocks, odd and even step counts, the deepest launch of each block size, several
launches, every precision, shift and coin kind, forward and adjoint.

Tolerance: a transform pair of length B commits at most 3u of the block's norm
per butterfly level and twiddle product (2 log2 B + 4 of them) and 4u for the
rounded matrices, so each launch adds at most (3 (2 * 13 + 4) + 4) u = 94u to an
amplitude of a normalised state; the oracle's own steps add 4u (double) each.
The float forms apply the coin rounded to float, as stepping does: 4u per step,
except for the Hadamard class, whose factor stays in double.
The double-float form rounds the stored state to 2^-47, bfloat16 to 2^-8."""
import numpy as np
import pytest

import oracle
from paper_1003_3779_gb300 import inputs
from tests.helpers import U, maxabs

pytestmark = pytest.mark.gpu

COINS = {"hadamard": inputs.hadamard(), "real": inputs.su2(0.3), "complex": inputs.su2(0.9, 0.4, -1.1)}


@pytest.fixture(scope="module")
def qw():
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    return qw


def tol(prec, T, launches, coin):
    u = U["f64"] if prec in ("f64", "comp") else U["f32"]
    store = {"comp": 2.0 ** -47, "bf16": 2.0 ** -8}.get(prec, 0.0)
    rounded = prec in ("f32", "bf16") and coin != "hadamard"
    return launches * (94 * u + store) + store + 4 * T * (u if rounded else U["f64"]) + 1e-15


def check(qw, n, T, prec, tile, k, coin="hadamard", shift=0, adjoint=False):
    C = COINS[coin]
    psi0 = inputs.random_state((2, n), seed=n + T)
    w = qw.Walk((n,), prec=prec, shift=shift).set_coin(C).set_plan_ex(k, tile, 2).set_state(psi0)
    assert w.plan_ex() == (k, tile, 2)
    w.set_clipping(False)
    want = oracle.evolve(psi0, C, T, shift=shift, adjoint=adjoint)
    (w.step_adjoint if adjoint else w.step)(T)
    assert maxabs(w.state(), want) <= tol(prec, T, -(-T // k) + 3, coin if shift == 0 else "")
    w.close()


@pytest.mark.parametrize("prec,tile", [("f32", 256), ("f32", 512), ("bf16", 256), ("bf16", 512), ("f64", 256), ("comp", 256)])
@pytest.mark.parametrize("n", [1, 2, 7, 2001, 8192, 20001])
def test_sizes_and_depths(qw, prec, tile, n):
    for T in (1, 2, 3, 64, 1365, 16 * tile - 1):
        check(qw, n, T, prec, tile, 16 * tile - 1)


@pytest.mark.parametrize("coin", list(COINS))
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("adjoint", [False, True])
def test_coins_shifts_and_directions(qw, coin, shift, adjoint):
    for prec, tile in (("f32", 256), ("f32", 512), ("f64", 256)):
        check(qw, 9001, 301, prec, tile, 150, coin, shift, adjoint)


def test_plan_is_checked(qw):
    w = qw.Walk((5000,), prec="f64").set_coin(inputs.hadamard())
    for k, tile in ((10, 512), (4096, 256), (0, 256), (10, 300)):
        with pytest.raises(qw.QWError):
            w.set_plan_ex(k, tile, 2)
    w.set_coin(2 * inputs.hadamard())       # not unitary
    with pytest.raises(qw.QWError):
        w.set_plan_ex(10, 256, 2)


def test_gain_left_by_stepping_is_applied(qw):
    """Stepping leaves rounded per-launch gains behind, which a following launch
    in momentum space takes up: the norm stays 1 to the float's accuracy."""
    n = 9001
    psi0 = inputs.random_state((2, n), seed=3)
    for C in (inputs.hadamard(), inputs.su2(0.3)):
        w = qw.Walk((n,), prec="f32").set_coin(C).set_plan_ex(64, 16, 1).set_state(psi0)
        w.step(2000)
        w.set_plan_ex(2000, 256, 2).step(2000)
        want = oracle.evolve(psi0, C, 4000)
        assert maxabs(w.state(), want) <= 4000 * 4 * U["f32"] / np.sqrt(n) + 94 * U["f32"]
        assert abs(w.norm() - 1) < 1e-6


def test_captured_calls_replay(qw):
    """A captured call recomputes its matrices on replay, so calls with other
    step counts in between do not disturb it."""
    import torch
    n, s = 30001, torch.cuda.Stream()
    psi0 = torch.from_numpy(inputs.random_state((2, n), seed=9)).to("cuda", torch.complex64)
    with torch.cuda.stream(s):
        w = qw.Walk((n,), prec="f32").set_coin(inputs.su2(0.7)).set_plan_ex(512, 256, 2).set_state(psi0)
        w.step(300)
        want = w.state()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            w.set_state(psi0)
            w.step(300)
        w.set_state(psi0).step(211).step(100)   # (two launches: the replay's buffer is the current one)
        g.replay()
        s.synchronize()
        assert np.array_equal(w.state(), want)
        w.set_state(psi0).step(211)
        a = w.state()
        w.set_plan_ex(512, 512, 2).set_plan_ex(512, 256, 2).set_state(psi0).step(211)
        assert np.array_equal(w.state(), a)
