"""qw_backward on a torus with more rows than a launch's second grid dimension
takes in tiles (65535 x 24 rows): against the oracle gradient.

Tolerance: a gradient entry is a sum over T steps of 2 Im(conj(a) b), |a| and |b|
at most the largest site norm A of any time (the walk mixes at most the four
neighbours, so A <= 4^t max |psi_0|; measured from the oracle's end states here and
doubled).  Each factor carries at most 2 T steps' rounding of 4u: the bound is
T * 2 * A^2 * 2 * (2 T * 4u)."""
import numpy as np
import pytest

import oracle
from paper_1003_3779_gb300 import inputs
from tests.helpers import U, maxabs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,shift", [("f32", 0), ("f64", 1)])
def test_tall_torus_against_oracle_gradient(prec, shift):
    import paper_1003_3779_gb300.qw as qw
    Lx, Ly, T, K = 2, 1_600_003, 6, 4
    rng = np.random.default_rng(12)
    phi = rng.uniform(-0.5, 0.5, size=(Ly, Lx, 4)).astype(np.float32).astype(np.float64)
    psi0 = (rng.standard_normal((4, Ly, Lx)) + 1j * rng.standard_normal((4, Ly, Lx))).astype(np.complex64)
    rect = (0, 5, 2, Ly - 9)
    _, want = oracle.region_grad(psi0, inputs.grover(), phi, T, rect, shift=shift, openmp=True)
    A = 2 * max(np.sqrt((np.abs(p) ** 2).sum(0).max())
                for p in (psi0, oracle.evolve(psi0, inputs.grover(), T, shift=shift, phi=phi.reshape(-1, 4), openmp=True)))
    w = qw.Walk((Lx, Ly), prec=prec, shift=shift).set_coin_phases(inputs.grover(), phi.reshape(-1, 4).astype(np.float32))
    w.set_state(psi0)
    grad = np.empty((Lx * Ly, 4))
    qw.qw_backward(w.h, rect, T, K, grad)
    assert maxabs(grad.reshape(Ly, Lx, 4), want) < 32 * T * T * U[prec] * A * A
    w.close()
