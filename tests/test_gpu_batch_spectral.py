"""Batches in momentum space (qw_batch_autotune) against the oracle and the
stepping variants: every transform length, T = 0, 1 and the longest, short
cycles that the cone goes round many times, odd and even, real, complex and
near-diagonal coins; exact zeros outside the cone and on the other parity;
repeated runs, plans set before and after.

Tolerance: the transform adds at most 3 (13 + 4) u and the factors 20 u of a
normalised state, 71u; the coin rounded to float 4u per step (amp_tol)."""
import numpy as np
import pytest

import oracle
from paper_1003_3779_gb300 import inputs
from tests.helpers import U, amp_tol, maxabs

pytestmark = pytest.mark.gpu

CS = inputs.BATCH_COIN_STATE


@pytest.fixture(scope="module")
def qw():
    import paper_1003_3779_gb300.qw as qw
    qw.lib()
    return qw


def oracle_walk(N, T, coin, x0, cs=CS):
    return oracle.evolve(inputs.localized_1d(N, x0, cs), coin, T)


def tuned(qw, N, T, coins, x0, cs=CS):
    b = qw.Batch(N, T, coins, x0, cs)
    rep = b.autotune()
    assert '"spectral": true' in rep, rep
    return b


@pytest.mark.parametrize("kind", ["real", "hadamard", "complex", "near_diagonal"])
def test_lengths_and_cycles(qw, kind):
    T = np.array([0, 1, 2, 255, 256, 511, 700, 1023, 1024, 2047, 3000, 4095, 4096, 8191] * 3)
    N = np.concatenate([np.full(14, 20011), np.array([1, 2, 3, 5, 64, 100, 101, 999, 1000, 2001, 2048, 513, 700, 30]),
                        np.array([7, 300, 2, 511, 513, 1023, 1401, 2048, 2049, 4096, 6001, 8192, 8193, 16384])])
    x0 = np.array([(31 * i * i + 7 * i) % n for i, n in enumerate(N)])
    x0[14:20] = np.minimum(N[14:20] - 1, x0[14:20])
    rng = np.random.default_rng(71)
    if kind == "near_diagonal":
        coins = np.stack([inputs.su2(t) for t in rng.choice([1e-4, np.pi / 2 - 1e-4, 0.0, np.pi / 2], len(N))])
    elif kind == "hadamard":
        coins = np.stack([inputs.hadamard()] * len(N))
    elif kind == "real":
        coins = np.stack([inputs.su2(t) for t in rng.uniform(0.1, 1.5, len(N))])
    else:
        coins = np.stack([inputs.random_unitary(2, rng) for _ in N])
    b = tuned(qw, N, T, coins, x0)
    for _ in range(2):                       # a second run starts again
        b.step()
        P, norms = b.probabilities()
        for i in range(len(N)):
            want = oracle_walk(int(N[i]), int(T[i]), coins[i], int(x0[i]))
            got = b.state(i)
            assert maxabs(got, want) < amp_tol("f32", int(T[i])) + 71 * U["f32"], i
            Pi = P[b.offsets[i]:b.offsets[i + 1]]
            assert np.abs(Pi - np.sum(np.abs(want) ** 2, axis=0)).sum() < 1e-4, i
            assert abs(norms[i] - Pi.astype(np.float64).sum()) < 1e-6
            d = (np.arange(N[i]) - x0[i]) % N[i]
            d = np.minimum(d, N[i] - d)
            if 2 * T[i] + 1 <= N[i]:
                assert np.all(Pi[(d > T[i]) | ((d - T[i]) % 2 != 0)] == 0.0)
    b.close()


def test_plans_take_over_and_back(qw):
    rng = np.random.default_rng(72)
    N, T = rng.integers(300, 9000, 200), rng.integers(64, 2000, 200)
    x0 = (rng.uniform(size=200) * N).astype(np.int64)
    coins = np.stack([inputs.su2(t) for t in rng.uniform(0.1, 1.4, 200)])
    b = tuned(qw, N, T, coins, x0, (0.6, 0.8j))
    P0 = b.step().probabilities()[0].copy()
    b.set_plan_ex(48, 1)                     # stepping again
    P1 = b.step().probabilities()[0].copy()
    assert np.abs(P0 - P1).max() < 2e-5
    rep = b.autotune()
    assert '"spectral": true' in rep
    assert np.array_equal(b.step().probabilities()[0], P0)
    b.set_cta_walks(0)
    assert np.abs(b.step().probabilities()[0] - P1).max() < 1e-6
    b.close()


def test_what_cannot_run_there_keeps_stepping(qw):
    N, x0 = np.array([20000, 3000]), np.array([10, 20])
    coins = np.stack([inputs.su2(0.4)] * 2)
    for T, c, prec in ((np.array([9000, 100]), coins, "f32"), (np.array([900, 100]), 0.9 * coins, "f32"),
                       (np.array([900, 100]), coins, "bf16"), (np.array([900, 100]), coins, "comp")):
        b = qw.Batch(N, T, c, x0, CS, prec=prec)
        assert '"spectral": true' not in b.autotune()
        b.step()
        b.close()
