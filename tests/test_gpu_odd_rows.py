"""Tori whose rows are no whole number of 16-byte vectors and at least one full
warp segment long, against the oracle: the 2D step kernels must not take the
alignment of one row for that of its neighbours.  Tolerance: amp_tol."""
import numpy as np
import pytest

import oracle
from paper_1003_3779_gb300 import inputs
from tests.helpers import amp_tol, maxabs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qw():
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    return qw


@pytest.mark.parametrize("prec,dims,k", [("f32", (129, 12), 1), ("f32", (301, 31), 4), ("f32", (301, 31), 8),
                                         ("f64", (129, 12), 1), ("comp", (129, 12), 1), ("bf16", (259, 12), 1),
                                         ("bf16", (258, 12), 1)])
@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("adjoint", [False, True])
def test_odd_rows(qw, prec, dims, k, shift, adjoint):
    Lx, Ly = dims
    T = 2 * k + 1
    psi0 = inputs.random_state((4, Ly, Lx), seed=31)
    want = oracle.evolve(psi0, inputs.grover(), T, shift=shift, adjoint=adjoint)
    w = qw.Walk(dims, prec=prec, shift=shift).set_coin(inputs.grover()).set_plan(k).set_state(psi0)
    (w.step_adjoint if adjoint else w.step)(T)
    assert maxabs(w.state(), want) < amp_tol(prec, T)
    w.close()


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_odd_rows_phase_coin(qw, prec):
    Lx, Ly, T = 131, 9, 5
    psi0 = inputs.random_state((4, Ly, Lx), seed=32)
    phi = np.random.default_rng(33).uniform(-0.5, 0.5, size=(Ly, Lx, 4)).astype(np.float32)
    B = inputs.grover()
    want = oracle.evolve(psi0, B, T, phi=phi.reshape(-1, 4).astype(np.float64))
    w = qw.Walk((Lx, Ly), prec=prec).set_coin_phases(B, phi.reshape(-1, 4)).set_state(psi0)
    assert maxabs(w.step(T).state(), want) < amp_tol(prec, T)
    w.close()
