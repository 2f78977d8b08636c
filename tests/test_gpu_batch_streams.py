"""A batch on a non-blocking stream, created, tuned and run without a pause: all of
its tables are in place when its kernels read them.  Tolerance as in
test_gpu_batch_spectral."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1003_3779_gb300 import inputs
from tests.helpers import U, amp_tol, maxabs

pytestmark = pytest.mark.gpu


def test_non_blocking_stream():
    import torch
    import paper_1003_3779_gb300.qw as qw
    s = torch.cuda.Stream()      # (torch's streams do not wait for the default stream)
    rng = np.random.default_rng(81)
    n = 3000
    N, T = rng.integers(300, 2000, n), rng.integers(64, 600, n)
    x0 = (rng.uniform(size=n) * N).astype(np.int64)
    theta = rng.uniform(0.1, 1.4, n)
    theta[::10] = 1e-4           # near-diagonal: stepped beside the transforms
    coins = np.stack([inputs.su2(t) for t in theta])
    for _ in range(2):
        b = qw.Batch(N, T, coins, x0, inputs.BATCH_COIN_STATE, stream=ctypes.c_void_p(s.cuda_stream))
        b.autotune()
        b.step()
        for i in (0, 1, 10, 1500, 1501, 2990, 2999):
            want = oracle.evolve(inputs.localized_1d(int(N[i]), int(x0[i]), inputs.BATCH_COIN_STATE), coins[i], int(T[i]))
            assert maxabs(b.state(i), want) < amp_tol("f32", int(T[i])) + 71 * U["f32"], i
        b.set_plan_ex(48, 1).step()
        P = b.probabilities()[0]
        for i in (0, 1, 2999):
            want = oracle.evolve(inputs.localized_1d(int(N[i]), int(x0[i]), inputs.BATCH_COIN_STATE), coins[i], int(T[i]))
            assert np.abs(P[b.offsets[i]:b.offsets[i + 1]] - (np.abs(want) ** 2).sum(0)).sum() < 1e-4
        b.close()
