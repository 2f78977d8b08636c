"""Calls captured into a CUDA graph do what they were captured for on every replay,
whatever else the handle did in between."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1003_3779_gb300 import inputs
from tests.helpers import U, amp_tol, maxabs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qw():
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    return qw


@pytest.mark.parametrize("dims", [(4096,), (96, 80)])
def test_captured_readout_reads_the_whole_state(qw, dims):
    """A readout captured while the state's box was small: replayed after more
    steps it gives every amplitude and probability of the wider state."""
    import torch
    s = torch.cuda.Stream()
    if len(dims) == 1:
        C, psi0 = inputs.su2(0.3), inputs.localized_1d(dims[0], 100)
    else:
        C, psi0 = inputs.grover(), inputs.localized_2d(dims[0], 30, 20, Ly=dims[1])
    psi = torch.from_numpy(psi0.astype(np.complex64)).cuda()
    w = qw.Walk(dims, prec="f32", stream=ctypes.c_void_p(s.cuda_stream)).set_coin(C)
    w.set_plan_ex(8, 16, 0) if len(dims) == 1 else w.set_plan(8)
    w.set_state(psi).step(8)
    out = torch.empty_like(psi)
    P = torch.empty(psi.shape[1:], dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        qw.qw_get_state(w.h, out)
        qw.qw_probabilities(w.h, P, want_norm=False)
    w.step(16)                        # two launches: the captured buffer is the current one again
    assert w.describe()["support"] != "full"
    with torch.cuda.stream(s):
        g.replay()
    torch.cuda.synchronize()
    want = oracle.evolve(psi0, C, 24)
    assert maxabs(out.cpu().numpy(), want) < amp_tol("f32", 24)
    assert maxabs(P.cpu().numpy(), (np.abs(want) ** 2).sum(0)) < 2 * amp_tol("f32", 24)
    w.close()


def test_captured_momentum_space_call_survives_another_tile(qw):
    """A momentum-space call captured with one tile, replayed after the handle ran
    with the other (tolerance: one launch, as in test_gpu_spectral)."""
    import torch
    n, s = 30001, torch.cuda.Stream()
    psi0 = inputs.random_state((2, n), seed=9)
    psi = torch.from_numpy(psi0).to("cuda", torch.complex64)
    C = inputs.su2(0.7)
    with torch.cuda.stream(s):
        for tile, other in ((256, 512), (512, 256)):
            w = qw.Walk((n,), prec="f32").set_coin(C).set_plan_ex(512, tile, 2).set_state(psi)
            w.step(300)
            want = w.state()
            assert maxabs(want, oracle.evolve(psi0, C, 300)) <= (300 * 4 / np.sqrt(n) + 94) * U["f32"]
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                w.set_state(psi)
                w.step(300)
            w.set_plan_ex(512, other, 2).set_state(psi).step(211).step(100)   # two launches: the captured buffers again
            g.replay()
            s.synchronize()
            assert np.array_equal(w.state(), want)
            w.close()
