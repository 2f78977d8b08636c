"""qw_describe's "kernel" names the kernel that the next forward step launches."""
import numpy as np
import pytest

from paper_1003_3779_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qw():
    import torch
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    launched(lambda: torch.zeros(1, device="cuda"))   # (a process's first profile may miss its kernels)
    return qw


def launched(fn):
    """Names of the step kernels that fn launches."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        fn()
        torch.cuda.synchronize()
    names = {e.name.split("<")[0].split("::")[-1].split("(")[0].split()[-1] for e in p.events()}
    return {n for n in names if n.startswith(("k_step", "k_tile"))}


CASES = {   # name: (dims, precision, boundary, shift, what else)
    "cycle sweep": ((5000,), "f32", 0, 0, ""), "cycle tiles": ((301,), "f32", 0, 0, ""), "cycle k1": ((5000,), "f32", 0, 0, "k1"),
    "cycle clipped": ((5000,), "f32", 0, 0, "site"), "cycle links": ((5000,), "f32", 0, 0, "links"),
    "segment": ((5000,), "f64", 1, 0, ""), "line wide": ((40000,), "f32", 2, 0, ""), "line clipped": ((40000,), "f32", 2, 0, "site"),
    "torus small": ((300, 200), "f32", 0, 0, ""), "torus large": ((1024, 768), "f32", 0, 0, ""),
    "torus clipped": ((1024, 768), "f32", 0, 0, "site"), "torus k1": ((300, 200), "f32", 0, 0, "k1"),
    "torus f64": ((300, 200), "f64", 0, 0, ""), "torus phases": ((300, 200), "f32", 0, 0, "phases"),
    "torus phases f64": ((300, 200), "f64", 0, 0, "phases"), "torus phases comp": ((60, 40), "comp", 0, 0, "phases"),
    "torus links": ((300, 200), "f32", 0, 0, "links"), "torus links f64": ((300, 200), "f64", 0, 0, "links"),
    "plane": ((300, 200), "f32", 1, 0, ""), "torus per site": ((30, 20), "f32", 0, 0, "per_site"),
    "torus complex": ((1024, 768), "f32", 0, 0, "complex"),
}


@pytest.mark.parametrize("name", list(CASES))
def test_kernel_is_the_one_that_runs(qw, name):
    dims, prec, bc, shift, what = CASES[name]
    d, ns = 2 * len(dims), int(np.prod(dims))
    rng = np.random.default_rng(6)
    w = qw.Walk(dims, prec=prec, bc=bc, shift=shift)
    base = inputs.hadamard() if d == 2 else inputs.grover()
    if what == "phases":
        w.set_coin_phases(base, rng.uniform(-1, 1, size=(ns, d)).astype(np.float32))
    elif what == "per_site":
        w.set_coin(np.stack([inputs.random_unitary(d, rng) for _ in range(ns)]), per_site=True)
    else:
        w.set_coin(inputs.random_unitary(d, rng) if what == "complex" else base)
    if what == "links":
        w.set_link_noise(0.1, 3)
    if what == "k1":
        w.set_plan(1)
    shape = (d,) + tuple(reversed(dims))
    if what == "site":
        psi0 = np.zeros(shape, complex)
        psi0[(0,) + tuple(n // 2 for n in shape[1:])] = 1
    else:
        psi0 = inputs.random_state(shape, seed=7)
    w.set_state(psi0).step(16)     # (the box of a localised state is known from here)
    assert launched(lambda: w.step(16)) == {w.describe()["kernel"]}
    w.close()
