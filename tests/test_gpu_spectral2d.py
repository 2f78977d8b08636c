"""GPU parity of the torus' momentum-space steps (qw_autotune) against the FP64
oracle and, on larger lattices, a complex128 evaluation in momentum space: every
transform length, cyclic axes and blocks with ragged ends, lattices smaller than
a block, odd and even step counts, several launches, the three shifts, both coins
of the path, forward and adjoint, and states at low momentum, where the matrices
are nearly degenerate.

Tolerance: a launch transforms twice each way over at most 13 + 12 butterfly levels
and 12 twiddle products at 3u of the norm each, and applies the matrix with 20u:
3 (2 * 25 + 12) u + 20 u = 206u per launch (of the norm, in norm); the oracle
adds 4u (double) per step, single steps 4u (float)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1003_3779_gb300 import inputs
from tests.helpers import U, maxabs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qw():
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    return qw


def exact(psi0, coin, T, shift, adjoint):
    """The same in complex128, by the matrix power of every momentum."""
    psi = torch.from_numpy(np.asarray(psi0, dtype=np.complex128)).cuda()
    _, ny, nx = psi.shape
    f = torch.fft.fft2(psi).permute(1, 2, 0).reshape(-1, 4, 1)
    ex = torch.exp(2j * np.pi * torch.arange(nx, dtype=torch.float64, device="cuda") / nx)[None, :].expand(ny, nx)
    ey = torch.exp(2j * np.pi * torch.arange(ny, dtype=torch.float64, device="cuda") / ny)[:, None].expand(ny, nx)
    ph = [ex.conj() * ey.conj(), ex.conj() * ey, ex * ey.conj(), ex * ey] if shift == 2 else [ex.conj(), ex, ey.conj(), ey]
    C = torch.from_numpy(coin).cuda()
    rows = [ph[c].reshape(-1, 1) * C[c] for c in range(4)]
    Um = torch.stack([rows[c ^ 1] if shift == 1 else rows[c] for c in range(4)], dim=1)
    if adjoint:
        Um = Um.conj().transpose(1, 2)
    out = torch.linalg.matrix_power(Um, T) @ f
    return torch.fft.ifft2(out.reshape(ny, nx, 4).permute(2, 0, 1)).cpu().numpy()


def check(qw, psi0, coin, T, shift=0, adjoint=False, force=True):
    _, ny, nx = psi0.shape
    w = qw.Walk((nx, ny), prec="f32", shift=shift).set_coin(coin).set_clipping(False).set_state(psi0)
    rep = w.autotune()
    if force:
        assert '"spectral"' in rep, rep
    (w.step_adjoint if adjoint else w.step)(T)
    want = exact(psi0, coin, T, shift, adjoint)
    err = np.sqrt(np.sum(np.abs(w.state() - want) ** 2)) / np.sqrt(np.sum(np.abs(want) ** 2))
    launches = 8
    assert err <= launches * 206 * U["f32"] + T * 4 * U["f64"]
    d = w.describe()
    w.close()
    return err, d


GROVER, HH = inputs.grover(), inputs.hadamard2()


@pytest.mark.parametrize("dims", [(256, 256), (512, 1024), (1024, 256), (2048, 512), (300, 200), (1000, 700), (257, 1025), (256, 8192),
                                  (300, 8192), (8192, 300)])
@pytest.mark.parametrize("coin,shift", [("grover", 0), ("grover", 1), ("grover", 2), ("hh", 2)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_sizes_shifts_and_directions(qw, dims, coin, shift, adjoint):
    psi0 = inputs.random_state((4, dims[1], dims[0]), seed=61)
    for T in (257, 300):
        err, d = check(qw, psi0, GROVER if coin == "grover" else HH, T, shift, adjoint)
        assert err < 2e-6       # (far inside the bound: the transforms' rms error)
        assert d["spectral"]["from_steps"] <= T


@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("k", [(0, 0), (1, 0), (1, 1), (128, 128), (127, 128), (128, 0), (64, 192), (3, 125)])
def test_single_momenta(qw, shift, k):
    """Plane waves, the nearly degenerate momenta among them: the error stays at
    the transforms' level, no factor of K."""
    n, T = 256, 1000
    y, x = np.mgrid[0:n, 0:n]
    wave = np.exp(2j * np.pi * (k[0] * x + k[1] * y) / n) / n
    v = np.array([0.6, -0.3 + 0.2j, 0.5j, 0.4])
    psi0 = (v / np.linalg.norm(v))[:, None, None] * wave
    err, _ = check(qw, psi0, GROVER, T, shift)
    assert err < 4e-6


def test_against_the_oracle_and_short_calls(qw):
    """A whole call against the oracle's steps; calls below the threshold step."""
    nx, ny, T = 300, 200, 301
    psi0 = inputs.random_state((4, ny, nx), seed=62)
    w = qw.Walk((nx, ny), prec="f32").set_coin(GROVER).set_state(psi0)
    w.autotune()
    w.step(T)
    assert maxabs(w.state(), oracle.evolve(psi0, GROVER, T, openmp=True)) < T * 4 * U["f32"]
    plan = w.plan_ex()
    w.set_state(psi0).step(9)
    v = qw.Walk((nx, ny), prec="f32").set_coin(GROVER).set_plan(plan[0]).set_state(psi0).step(9)
    assert np.array_equal(w.state(), v.state())
    # a localised state is stepped while its box grows
    psi1 = inputs.localized_2d(nx, 150, 100, Ly=ny)
    w.set_state(psi1).step(90)
    v.set_state(psi1).step(90)
    assert np.array_equal(w.state(), v.state())


def test_a_plan_set_after_autotune_steps(qw):
    """qw_set_plan takes the momentum-space steps back: the same bits as the plan
    on a handle that was never tuned."""
    psi0 = inputs.random_state((4, 128, 128), seed=4, dtype=np.complex64)
    w = qw.Walk((128, 128), prec="f32").set_coin(inputs.grover()).set_state(psi0)
    w.autotune()
    w.set_plan(8)
    v = qw.Walk((128, 128), prec="f32").set_coin(inputs.grover()).set_plan(8)
    assert "spectral" not in w.describe()
    assert np.array_equal(w.set_state(psi0).step(200).state(np.complex64), v.set_state(psi0).step(200).state(np.complex64))
    w.close()
    v.close()
