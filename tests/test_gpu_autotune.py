"""What qw_autotune settles on: never a plan that it did not time against the
kernels that the steps then run, whatever was tuned or cached before."""
import json
import os
import subprocess
import sys
import time

import numpy as np
import pytest

from paper_1003_3779_gb300 import inputs

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


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


def tuned(code, env=None):
    """Run `code` in a process of its own; the JSON lines it prints."""
    head = "import json, numpy as np\nfrom paper_1003_3779_gb300 import inputs, qw\n"
    p = subprocess.run([sys.executable, "-c", head + code], cwd=ROOT, env=dict(os.environ, **(env or {})),
                       capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stderr[-2000:]
    return [json.loads(line) for line in p.stdout.splitlines()]


TUNE = """
def tune(coin):
    w = qw.Walk((1 << 20,), prec="f32").set_coin(coin).set_state(inputs.random_state((2, 1 << 20), seed=1))
    print(w.autotune())
    w.close()
"""


def test_a_cache_of_stepping_plans_gets_the_momentum_space_form(qw, tmp_path):
    """A tuning file that holds the stepping plan alone: the momentum-space form is
    timed against that plan, used, and added to the file."""
    path = tmp_path / "tune.json"
    env = {"QW_TUNE_CACHE": str(path)}
    (first,) = tuned(TUNE + "tune(inputs.su2(0.3))\n", env)
    assert not first["cached"] and "spectral" in first
    path.write_text("".join(line for line in path.read_text().splitlines(True) if "_spectral" not in line))
    (again,) = tuned(TUNE + "tune(inputs.su2(0.3))\n", env)
    assert again["cached"] and again["spectral"]["from_steps"] >= 1
    assert "_spectral" in path.read_text()


def test_a_coin_that_is_not_unitary_tuned_first(qw):
    lossy, unitary = tuned(TUNE + "tune(0.9 * inputs.su2(0.3))\ntune(inputs.su2(0.3))\n")
    assert "spectral" not in lossy and unitary["cached"] and "spectral" in unitary


def test_a_failed_allocation_is_not_remembered(qw):
    """No room for the tables of one handle: it steps; the next one, with room,
    takes the momentum-space form."""
    code = """
import os
w = [qw.Walk((1 << 20,), prec="f32").set_coin(inputs.su2(0.3)).set_state(inputs.random_state((2, 1 << 20), seed=1)) for _ in range(2)]
w[0].step(1)
os.environ["QW_FAULT"] = "alloc"
qw.lib()
print(w[0].autotune())
del os.environ["QW_FAULT"]
print(w[1].autotune())
"""
    starved, fed = tuned(code)
    assert starved["tuned"] and "spectral" not in starved and "spectral" in fed


def test_a_rejected_workspace_is_given_back(qw):
    """Two sites in x: a block of the transforms holds 128 times the lattice, so the
    torus goes on being stepped, and keeps none of the transforms' 77 MB."""
    import torch
    used = []
    for _ in range(2):      # (the first handle loads the kernels)
        w = qw.Walk((2, 300000), prec="f32").set_coin(inputs.grover()).set_state(
            inputs.random_state((4, 300000, 2), seed=2))
        w.step(1)
        w.synchronize()
        before = torch.cuda.mem_get_info()[0]
        assert "spectral" not in w.autotune()
        used.append(before - torch.cuda.mem_get_info()[0])
        w.close()
    assert used[1] < 16 << 20


@pytest.mark.parametrize("nx,ny,T", [(300, 200, 300000), (256, 256, 300000)])
def test_long_calls_stay_in_momentum_space(qw, nx, ny, T):
    """Calls of more steps than 64 of the longest launches: less than half the time
    of stepping them (a tenth to a third is expected)."""
    w = qw.Walk((nx, ny), prec="f32").set_coin(inputs.grover()).set_state(inputs.random_state((4, ny, nx), seed=3))
    assert '"spectral"' in w.autotune()
    v = qw.Walk((nx, ny), prec="f32").set_coin(inputs.grover()).set_plan(8).set_state(inputs.random_state((4, ny, nx), seed=3))
    took = []
    for walk in (w, v):
        walk.step(T).synchronize()
        t = time.perf_counter()
        walk.step(T).synchronize()
        took.append(time.perf_counter() - t)
        assert abs(walk.norm() - 1) < 1e-3
        walk.close()
    assert took[0] < 0.5 * took[1]


@pytest.mark.parametrize("nx,ny", [(300, 200), (700, 1100)])
def test_short_calls_leave_stepping_as_soon_as_they_gain(qw, nx, ny):
    """Calls of 64 steps take half the time in momentum space on these tori, where a
    call of 256 steps takes two launches or deeper halos."""
    w = qw.Walk((nx, ny), prec="f32").set_coin(inputs.grover()).set_state(inputs.random_state((4, ny, nx), seed=9))
    w.autotune()
    assert w.describe()["spectral"]["from_steps"] <= 80
    w.close()
