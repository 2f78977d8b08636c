"""What qw_autotune settles on: never a plan that it did not time against the
kernels that the steps then run, whatever was tuned or cached before."""
import numpy as np
import pytest

from paper_1003_3779_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qw():
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    return qw


@pytest.mark.parametrize("nx,ny", [(300, 200), (1024, 1024)])
def test_phase_coins_keep_several_steps_per_launch(qw, nx, ny):
    """A phase-coin torus runs in tiles, 2 to 6 times faster per step at k = 8 than
    a step per launch; the steps give the same bits, tuned or not."""
    phi = np.random.default_rng(3).uniform(-0.5, 0.5, size=(nx * ny, 4)).astype(np.float32)
    psi0 = inputs.random_state((4, ny, nx), seed=5, dtype=np.complex64)
    w = qw.Walk((nx, ny), prec="f32").set_coin_phases(inputs.grover(), phi).set_state(psi0)
    v = qw.Walk((nx, ny), prec="f32").set_coin_phases(inputs.grover(), phi).set_state(psi0)
    assert w.plan()[0] == 8
    w.autotune()
    assert w.plan()[0] > 1
    assert np.array_equal(w.set_state(psi0).step(21).state(np.complex64), v.step(21).state(np.complex64))
    w.close()
    v.close()


@pytest.mark.parametrize("shift", [0, 1, 2])
def test_general_coins_keep_several_steps_per_launch(qw, shift):
    """A general coin: tiles on a torus this small, whatever its class."""
    C = np.linalg.qr(np.random.default_rng(4).standard_normal((4, 4)))[0].astype(complex)
    psi0 = inputs.random_state((4, 200, 300), seed=6, dtype=np.complex64)
    w = qw.Walk((300, 200), prec="f32", shift=shift).set_coin(C).set_state(psi0)
    v = qw.Walk((300, 200), prec="f32", shift=shift).set_coin(C).set_state(psi0)
    assert v.plan()[0] == 8
    w.autotune()
    assert w.plan()[0] > 1
    w.set_plan(8)
    assert np.array_equal(w.set_state(psi0).step(21).state(np.complex64), v.step(21).state(np.complex64))
    w.close()
    v.close()
