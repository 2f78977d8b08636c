"""Phase coins on the torus: several steps per launch in tiles round as one step per
launch does, bit for bit, whatever the base coin's class."""
import numpy as np
import pytest

from paper_1003_3779_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coin", ["grover", "hh", "real", "complex"])
@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("start", ["dense", "site"])
def test_bits_of_single_steps(coin, shift, start):
    import paper_1003_3779_gb300.qw as qw
    Lx, Ly, T = 90, 71, 43
    rng = np.random.default_rng(21)
    C = {"grover": inputs.grover(), "hh": inputs.hadamard2(), "complex": inputs.random_unitary(4, rng),
         "real": np.linalg.qr(rng.standard_normal((4, 4)))[0].astype(complex)}[coin]
    phi = rng.uniform(-3, 3, size=(Lx * Ly, 4)).astype(np.float32)
    psi0 = inputs.random_state((4, Ly, Lx), seed=22) if start == "dense" else inputs.localized_2d(Lx, 40, 3, Ly=Ly)
    got = []
    for k in (8, 1):
        w = qw.Walk((Lx, Ly), prec="f32", shift=shift).set_coin_phases(C, phi).set_plan(k).set_state(psi0)
        got.append(w.step(T).state())
        w.close()
    assert np.array_equal(*got)
