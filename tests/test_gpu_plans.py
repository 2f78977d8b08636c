"""The plan a walk has without being told."""
import numpy as np
import pytest

from paper_1003_3779_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1 << 20, 16), (16, 1 << 18)])
def test_long_thin_tori_take_the_streaming_kernel(nx, ny):
    """Enough warps for the streaming kernel in one direction alone: eight steps
    per launch, with the bits of single steps."""
    import paper_1003_3779_gb300.qw as qw
    psi0 = inputs.random_state((4, ny, nx), seed=4, dtype=np.complex64)
    w = qw.Walk((nx, ny), prec="f32").set_coin(inputs.grover()).set_state(psi0)
    v = qw.Walk((nx, ny), prec="f32").set_coin(inputs.grover()).set_plan(1).set_state(psi0)
    assert w.plan()[0] == 8
    assert np.array_equal(w.step(20).state(np.complex64), v.step(20).state(np.complex64))
    w.close()
    v.close()
