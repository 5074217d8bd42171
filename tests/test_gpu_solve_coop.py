"""The one-launch conjugate-gradient solve (FP32, up to four right-hand sides)
over the sizes at which its work is cut: rows a block owns (n over the SM
count), row groups of 32 / columns, chunks of 4096 points, and their
remainders (GPU, C ABI).

The true FP64 residual of the returned W is at most 5 times the tolerance of
the recurrence, as the FP32 case of tests/test_gpu_solve.py asks; the
iteration count is the oracle's within max(3, 15%), and the columns are those
of the same system solved with more right-hand sides at once (the form with a
launch per step) to the tolerance."""
import numpy as np
import pytest
import torch

import synth
from _helpers import dev, host
from oracle import solve

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ab():
    import paper_1704_08907_gb300 as ab
    return ab


@pytest.mark.parametrize("n,nrhs", [(1, 1), (2, 3), (37, 4), (153, 1), (1001, 2), (1500, 3),
                                    (4096, 1), (4097, 4), (5000, 1)])
def test_against_fp64_and_the_stepwise_form(ab, cuda, n, nrhs):
    ctx = ab.Context(0)
    X = synth.uniform_positions(n, 3, 300 + n)
    rng = np.random.default_rng(301 + n)
    B = rng.standard_normal((n, 6)).astype(np.float32)
    A = solve.system_matrix(X[:, :3], 50.0, 0.25)
    tol = 1e-5
    W, it, rr = ab.ab_kernel_solve(ctx, dev(X), dev(B[:, :nrhs].copy()), 50.0, 0.25, "fp32", tol, 1000)
    ab.ab_sync(ctx)
    Wh = host(W).astype(np.float64)
    Bh = B[:, :nrhs].astype(np.float64)
    true = np.linalg.norm(Bh - A @ Wh, axis=0) / np.linalg.norm(Bh, axis=0)
    assert rr <= tol and true.max() <= 5 * tol
    _, it_ref, _ = solve.cg(X[:, :3], B[:, :nrhs], 50.0, 0.25, tol, 1000, A=A)
    assert abs(it - it_ref) <= max(3, 0.15 * it_ref)
    W6, _, _ = ab.ab_kernel_solve(ctx, dev(X), dev(B), 50.0, 0.25, "fp32", tol, 1000)
    # both within tol ||b|| / sigma^2 of the solution
    diff = np.linalg.norm(host(W6)[:, :nrhs] - Wh, axis=0)
    assert np.all(diff <= 2 * 5 * tol / 0.25 * np.linalg.norm(Bh, axis=0))
    again, it2, _ = ab.ab_kernel_solve(ctx, dev(X), dev(B[:, :nrhs].copy()), 50.0, 0.25, "fp32", tol, 1000)
    assert it2 == it and torch.equal(again, W)
    ctx.close()


def test_zero_column_and_iteration_limit(ab, cuda):
    ctx = ab.Context(0)
    n = 700
    X = dev(synth.uniform_positions(n, 3, 9))
    B = np.random.default_rng(10).standard_normal((n, 3)).astype(np.float32)
    B[:, 1] = 0.0
    W, it, rr = ab.ab_kernel_solve(ctx, X, dev(B), 50.0, 0.25, "fp32", 1e-5, 1000)
    assert torch.all(W[:, 1] == 0) and rr <= 1e-5 and it > 0
    W, it, rr = ab.ab_kernel_solve(ctx, X, dev(B), 50.0, 0.25, "fp32", 1e-5, 4)
    assert it == 4 and rr > 1e-5
    W, it, rr = ab.ab_kernel_solve(ctx, X, dev(B), 50.0, 0.25, "fp32", 1e-5, 0)
    assert it == 0 and torch.all(W == 0) and abs(rr - 1.0) < 1e-6
    W, it, rr = ab.ab_kernel_solve(ctx, X, dev(np.zeros((n, 1), np.float32)), 50.0, 0.25, "fp32", 1e-5, 10)
    assert it == 0 and torch.all(W == 0) and rr == 0.0
    ab.ab_sync(ctx)
    ctx.close()
