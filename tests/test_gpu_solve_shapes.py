"""Kernel-system solve on odd sizes: n * nrhs odd, where the workspace's FP64
partials follow vectors of an odd number of floats (GPU, C ABI)."""
import numpy as np
import pytest

import synth
from _helpers import dev, host
from oracle import solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nrhs", [(1001, 5), (333, 7), (9731, 1)])
def test_odd_sizes(cuda, n, nrhs):
    import paper_1704_08907_gb300 as ab
    ctx = ab.Context(0)
    X = synth.uniform_positions(n, 3, 500 + n)
    B = np.random.default_rng(501 + n).standard_normal((n, nrhs)).astype(np.float32)
    tol = 1e-4
    W, it, rr = ab.ab_kernel_solve(ctx, dev(X), dev(B), 200.0, 0.5, "fp32", tol, 1000)
    ab.ab_sync(ctx)
    A = solve.system_matrix(X[:, :3], 200.0, 0.5)
    Wh = host(W).astype(np.float64)
    true = np.linalg.norm(B - A @ Wh, axis=0) / np.linalg.norm(B, axis=0)
    assert it > 0 and rr <= tol and true.max() <= 5 * tol
    ctx.close()
