"""The gradient's backward sweep runs on the intersection of two light cones:
against the oracle for starts and regions that meet late, never, at both ends of
the torus or at once, checkpoint segments of every kind, both shifts, with and
without the known support of the start.  Tolerances as in test_gpu_backward."""
import numpy as np
import pytest

import oracle
from paper_1003_3779_gb300 import inputs
from tests.helpers import maxabs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qw():
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    return qw


@pytest.mark.parametrize("start,rect", [((0, 0), (12, 10, 4, 3)), ((30, 2), (0, 0, 5, 5)), ((24, 20), (22, 18, 6, 6)),
                                        ((3, 37), (40, 0, 8, 2)), ((10, 10), (5, 5, 0, 4)), ("dense", (7, 30, 9, 10)),
                                        ("corners", (20, 20, 2, 2))])
@pytest.mark.parametrize("T,K", [(5, 2), (17, 17), (40, 8), (61, 64)])
@pytest.mark.parametrize("prec,shift", [("f64", 0), ("f64", 1), ("f32", 0)])
def test_cones_against_oracle(qw, start, rect, T, K, prec, shift):
    Lx, Ly = 48, 41
    phi = np.random.default_rng(5).uniform(-0.5, 0.5, size=(Ly, Lx, 4)).astype(np.float32).astype(np.float64)
    if start == "dense":
        psi0 = inputs.random_state((4, Ly, Lx), seed=6)
    elif start == "corners":    # a support whose box is the whole torus
        psi0 = (inputs.localized_2d(Lx, 0, 0, Ly=Ly) + inputs.localized_2d(Lx, Lx - 1, Ly - 1, Ly=Ly)) / np.sqrt(2)
    else:
        psi0 = inputs.localized_2d(Lx, *start, Ly=Ly)
    want_loss, want = oracle.region_grad(psi0, inputs.grover(), phi, T, rect, shift=shift)
    for clip in (True, False):
        w = qw.Walk((Lx, Ly), prec=prec, shift=shift).set_clipping(clip)
        w.set_coin_phases(inputs.grover(), phi.reshape(-1, 4).astype(np.float32)).set_state(psi0)
        grad = np.full((Lx * Ly, 4), np.nan)
        loss = qw.qw_backward(w.h, rect, T, K, grad)
        tol = 1e-12 if prec == "f64" else 2e-5
        assert abs(loss - want_loss) < tol
        assert maxabs(grad.reshape(Ly, Lx, 4), want) < tol * max(1.0, np.abs(want).max())
        assert maxabs(w.state(), oracle.evolve(psi0, inputs.grover(), T, shift=shift, phi=phi.reshape(-1, 4))) < tol
        w.close()
