"""The solve's per-column scalars, written by one kernel and read by the next
while both are resident: many columns that stop after different numbers of
iterations, over several row blocks an SM, repeated (GPU, C ABI).

The true FP64 residual of every column is at most 5 times the tolerance of the
recurrence, as in tests/test_gpu_solve.py, and every repeat gives the same
bits: a stale step length would fail either."""
import numpy as np
import pytest
import torch

import synth
from _helpers import dev, host
from oracle import solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nrhs", [(2003, 63), (3001, 37)])
def test_columns_keep_their_own_steps(cuda, n, nrhs):
    import paper_1704_08907_gb300 as ab
    ctx = ab.Context(0)
    X = synth.uniform_positions(n, 3, 700 + n)
    A = solve.system_matrix(X[:, :3], 50.0, 0.25)
    B = np.random.default_rng(701 + n).standard_normal((n, nrhs))
    for c in range(0, nrhs, 3):      # smooth columns: fewer iterations
        B[:, c] = (A @ B[:, c]) * 10.0 ** (c % 7 - 3)
    B = B.astype(np.float32)
    tol = 1e-4
    W, it, rr = ab.ab_kernel_solve(ctx, dev(X), dev(B), 50.0, 0.25, "fp32", tol, 1000)
    ab.ab_sync(ctx)
    Wh = host(W).astype(np.float64)
    true = np.linalg.norm(B - A @ Wh, axis=0) / np.linalg.norm(B, axis=0)
    assert rr <= tol and true.max() <= 5 * tol
    for _ in range(5):
        again, it2, _ = ab.ab_kernel_solve(ctx, dev(X), dev(B), 50.0, 0.25, "fp32", tol, 1000)
        assert it2 == it and torch.equal(again, W)
    ab.ab_sync(ctx)
    ctx.close()
