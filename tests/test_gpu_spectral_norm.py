"""A momentum-space launch keeps the norm: rounding errors of single amplitudes average
out over a state, what is left of them below one rounding (u) of the norm per launch.
A systematic error of the transforms' constants or tables would not average out."""
import numpy as np
import pytest

from paper_1003_3779_gb300 import inputs
from tests.helpers import U

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qw():
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    return qw


@pytest.mark.parametrize("n,shift,coin", [(256, 0, "grover"), (512, 1, "grover"), (1024, 2, "hh"), (2048, 0, "grover")])
def test_torus(qw, n, shift, coin):
    psi0 = inputs.random_state((4, n, n), seed=11, dtype=np.complex64)
    w = qw.Walk((n, n), prec="f32", shift=shift).set_coin(inputs.grover() if coin == "grover" else inputs.hadamard2()).set_state(psi0)
    assert '"spectral"' in w.autotune()
    before = w.norm()
    assert abs(w.step(200).norm() - before) < U["f32"]      # (cyclic axes: one launch)
    w.close()


@pytest.mark.parametrize("tile,K", [(256, 512), (512, 1000)])
@pytest.mark.parametrize("theta", [0.3, np.pi / 4])
def test_cycle(qw, tile, K, theta):
    n = 1 << 20
    psi0 = inputs.random_state((2, n), seed=12, dtype=np.complex64)
    w = qw.Walk((n,), prec="f32").set_coin(inputs.su2(theta)).set_plan_ex(K, tile, 2).set_state(psi0)
    before = w.norm()
    assert abs(w.step(K).norm() - before) < U["f32"]
    w.close()
