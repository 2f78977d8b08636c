"""Clipped steps have the bits of stepping the whole cycle whatever plan it has: the
default, the tuned one, sweeps deeper than the warp tiles that windows run.  (Not
sweeps of more than 8 steps per site of a tile's lane in bf16 storage, which rounds the
state after every launch.)"""
import numpy as np
import pytest

from paper_1003_3779_gb300 import inputs

pytestmark = pytest.mark.gpu

COINS = {"hadamard": inputs.hadamard(), "signs": np.array([[-1, 1], [1, 1]]) / np.sqrt(2), "real": inputs.su2(0.3),
         "complex": inputs.su2(0.3, 0.4, -0.7)}


@pytest.fixture(scope="module")
def qw():
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    return qw


def both(qw, N, prec, coin, shift, adjoint, chunks, plan=None):
    got = []
    for clip in (True, False):
        w = qw.Walk((N,), prec=prec, shift=shift).set_coin(COINS[coin]).set_clipping(clip)
        if plan:
            w.set_plan_ex(*plan)
        w.set_state(inputs.localized_1d(N, N // 3, (0.6, 0.8j)))
        for T in chunks:
            (w.step_adjoint if adjoint else w.step)(T)
        got.append((w.state(), w.norm()))
        w.close()
    assert np.array_equal(got[0][0], got[1][0])
    assert abs(got[0][1] - 1) < (1e-12 if prec == "f64" else 1e-5 if prec == "f32" else 0.5)


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("coin", list(COINS))
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("N,chunks", [(40000, [1500]), (40000, [333, 7, 70]), (3001, [40, 300, 1700])])
def test_default_plan(qw, prec, coin, shift, adjoint, N, chunks):
    both(qw, N, prec, coin, shift, adjoint, chunks)


@pytest.mark.parametrize("prec,plan", [("f32", (510, 32, 1)), ("f32", (384, 32, 1)), ("f32", (200, 16, 1)), ("f32", (129, 16, 1)),
                                       ("f32", (37, 16, 1)), ("f64", (7, 8, 1)), ("f64", (20, 8, 1)), ("f64", (64, 8, 1)),
                                       ("f64", (101, 8, 1)), ("bf16", (100, 16, 1))])
@pytest.mark.parametrize("coin", list(COINS))
@pytest.mark.parametrize("N", [40000, 3001])
def test_sweeps_of_any_depth(qw, prec, plan, coin, N):
    both(qw, N, prec, coin, 0, False, [1001, 450, 100], plan)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("coin", list(COINS))
def test_tuned_plan(qw, prec, coin):
    """The tuned plan of a handle, clipped, against that plan set by hand, unclipped
    (a tuned handle's long calls on whole lattices leave stepping)."""
    N, T = 20000, 1111
    psi0 = inputs.localized_1d(N, 500, (0.6, 0.8j))
    w = qw.Walk((N,), prec=prec).set_coin(COINS[coin]).set_state(inputs.random_state((2, N), seed=8))
    w.autotune()
    v = qw.Walk((N,), prec=prec).set_coin(COINS[coin]).set_clipping(False).set_plan_ex(*w.plan_ex())
    assert np.array_equal(w.set_state(psi0).step(T).state(), v.set_state(psi0).step(T).state())
    w.close()
    v.close()


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("scale", [0.97, 1.01])
def test_coins_of_the_class_that_are_not_unitary(qw, prec, scale):
    """A factor per launch that is no power of two and, rounded to float, alternates."""
    N, got = 9000, []
    for clip in (True, False):
        w = qw.Walk((N,), prec=prec).set_coin(scale * inputs.hadamard()).set_clipping(clip)
        w.set_state(inputs.localized_1d(N, N // 3, (0.6, 0.8j)))
        for T in (300, 5, 12, 20, 70, 127, 129, 200):
            w.step(T)
        got.append(w.state())
        w.close()
    assert np.array_equal(*got)


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("coin", list(COINS))
@pytest.mark.parametrize("adjoint", [False, True])
def test_short_calls(qw, prec, coin, adjoint):
    both(qw, 3000, prec, coin, 0, adjoint, [5, 12, 20, 50, 70, 100, 127, 200])
