"""State in and out of a walk on the GPU: the copy that also searches the
support box, the box-limited readout and marginals, and the clearing of the
other buffer by the box of the previous run.  Copies are compared bit for bit,
walks with those of a fresh handle that steps the whole lattice."""
import numpy as np
import pytest
import torch

from paper_1003_3779_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qw():
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    return qw


def make(qw, dims, prec, **kw):
    coin = inputs.hadamard() if len(dims) == 1 else inputs.grover()
    return qw.Walk(dims, prec=prec, **kw).set_coin(coin)


DTYPE = {"f32": torch.complex64, "bf16": torch.complex64, "f64": torch.complex128, "comp": torch.complex128}


@pytest.mark.parametrize("prec", ["f32", "f64", "bf16", "comp"])
@pytest.mark.parametrize("dims", [(1,), (3,), (255,), (1000,), (100003,), (1, 7), (7, 1), (33, 5), (64, 48), (301, 211)])
@pytest.mark.parametrize("offset", [0, 1])
def test_round_trip_and_support(qw, prec, dims, offset):
    shape = (2 * len(dims),) + tuple(reversed(dims))
    n = int(np.prod(shape))
    rng = np.random.default_rng(n)
    sites = [tuple(int(rng.integers(0, s)) for s in shape[1:]) for _ in range(2)]
    for where in (sites[:1], sites, [tuple(s - 1 for s in shape[1:])]):
        # offset 1: a buffer that starts one amplitude after a 16-byte boundary
        psi = torch.zeros(n + offset, dtype=DTYPE[prec], device="cuda")[offset:].view(shape)
        for i, s in enumerate(where):
            psi[(i % shape[0],) + s] = 0.5 - 0.25j * i
        w = make(qw, dims, prec).set_state(psi)
        out = torch.empty(n + offset, dtype=DTYPE[prec], device="cuda")[offset:].view(shape)
        assert torch.equal(qw.qw_get_state(w.h, out), psi)
        w.step(1)                              # resolves the box, which then grows by one
        w.step_adjoint(1)
        lo = [min(s[a] for s in where) for a in range(len(dims))]
        hi = [max(s[a] for s in where) for a in range(len(dims))]
        want = []
        for a in reversed(range(len(dims))):   # columns first
            L, b0, bw = shape[1 + a], lo[a] - 2, hi[a] - lo[a] + 5
            want += [0, L] if bw >= L else [b0 % L, bw]
        want = (want + [0, 1])[:4]
        full = want[1] == shape[-1] and (len(dims) == 1 or want[3] == shape[1])
        assert w.describe()["support"] == ("full" if full else want)
        P = torch.empty(shape[1:], dtype=torch.float32, device="cuda")
        qw.qw_probabilities(w.h, P, want_norm=False)
        qw.qw_get_state(w.h, out)
        ref = (out.abs().double() ** 2).sum(0)
        assert float((P.double() - ref).abs().max()) <= 2.0 ** -22
        w.close()


@pytest.mark.parametrize("dims,bc", [((4001,), 0), ((4001,), 2), ((300, 170), 0), ((300, 170), 1)])
@pytest.mark.parametrize("prec", ["f32", "f64", "bf16", "comp"])
def test_reused_handle_equals_a_fresh_one(qw, dims, bc, prec):
    """Runs from different sites on one handle: what an earlier run left in the
    buffers (clipped, over the whole lattice, tuned, or by a graph replay) does
    not reach the next one."""
    L = dims[0]

    def start(x, y):
        return inputs.localized_1d(L, x) if len(dims) == 1 else inputs.localized_2d(L, x, y, Ly=dims[1])

    def fresh(psi, T):
        w = make(qw, dims, prec, bc=bc).set_state(psi)
        out = w.step(T).state()
        w.close()
        return out

    w = make(qw, dims, prec, bc=bc)
    dev = torch.from_numpy(start(5, 3)).to("cuda", DTYPE[prec])
    for i, (x, y, T) in enumerate([(L // 2, 80, 20), (3, 1, 33), (L - 2, 150, 7), (40, 40, 12), (200, 9, 25)]):
        psi = start(x, y)
        if i == 3:                             # a dense run in between
            w.set_state(inputs.random_state((2 * len(dims),) + tuple(reversed(dims)), seed=1)).step(9)
        if i == 4:                             # the tuner writes the other buffer
            w.set_state(psi).step(3)
            plan = w.plan_ex()
            w.autotune()
            w.set_plan_ex(*plan) if len(dims) == 1 and bc == 0 else None
            if len(dims) == 2:
                w.set_plan(0)
        w.set_state(torch.from_numpy(psi).to("cuda", DTYPE[prec]) if i % 2 else psi)
        got, want = w.step(T).state(), fresh(psi, T)
        if i < 4:                              # (the default plan is not the tuned one: same to rounding)
            assert np.array_equal(got, want)
        assert np.abs(got - want).max() < (1e-5 if prec != "bf16" else 0.1)
    # a captured run of a dense state leaves both buffers full behind the host's back
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        w2 = make(qw, dims, prec, bc=bc, stream=None)
        dense = torch.from_numpy(inputs.random_state((2 * len(dims),) + tuple(reversed(dims)), seed=2)).to("cuda", DTYPE[prec])
        w2.set_state(dense).step(3)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            w2.set_state(dense)
            w2.step(3)
        w2.set_state(dev).step(4)
        g.replay()
        w2.set_state(dev).step(11)
        got = w2.state()
        s.synchronize()
        w2.close()
    assert np.array_equal(got, fresh(dev.cpu().numpy(), 11))
    w.close()


@pytest.mark.parametrize("dims", [(1 << 20,), (1000003,), (1024, 1024), (4096, 512)])
@pytest.mark.parametrize("prec,dtype", [("f64", torch.complex64), ("comp", torch.complex64), ("f32", torch.complex128),
                                        ("bf16", torch.complex64)])
def test_dense_states_fill_the_box(qw, dims, prec, dtype):
    """Converted states are searched in the buffer, by blocks that stop once the
    box is full, while others still add to it: the box is the whole lattice, and
    every run of the same state ends in the same bits."""
    g = torch.Generator(device="cuda").manual_seed(len(dims))
    psi = torch.randn((2 * len(dims),) + tuple(reversed(dims)), dtype=dtype, device="cuda", generator=g)
    psi /= psi.abs().square().sum().sqrt()
    w, first = make(qw, dims, prec), None
    for _ in range(25):
        w.set_state(psi).step(3)
        assert w.describe()["support"] == "full"
        out = qw.qw_get_state(w.h, torch.empty_like(psi))
        first = out if first is None else first
        assert torch.equal(out, first)
    w.close()
