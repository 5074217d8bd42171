"""A one-launch solve whose waits run out: the call itself reports the timeout
(it has synchronised), reports no residual that could pass for convergence,
leaves no error for ab_sync, and the next solve is that of a fresh context bit
for bit (GPU, C ABI).  One block takes no part; the others' first wait gives
up after 20 ms."""
import numpy as np
import pytest
import torch

import synth
from _helpers import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nrhs,absent", [(1, 1, 0), (1000, 1, 0), (1000, 3, 7), (4096, 2, 127)])
def test_timeout_is_reported_by_the_call(cuda, n, nrhs, absent):
    import paper_1704_08907_gb300 as ab
    ctx = ab.Context(0)
    X = dev(synth.uniform_positions(n, 3, 800 + n))
    B = dev(np.random.default_rng(801 + n).standard_normal((n, nrhs)).astype(np.float32))
    W, it, rr = ab.ab_kernel_solve(ctx, X, B, 50.0, 0.25, "fp32", 1e-4, 1000)
    assert rr <= 1e-4
    ab.ab_testing_solve_timeout(ctx, absent, 20_000_000)
    with pytest.raises(ab.AbError) as e:
        ab.ab_kernel_solve(ctx, X, B, 50.0, 0.25, "fp32", 1e-4, 1000)
    assert e.value.status == ab._abi.AB_ERR_TIMEOUT
    ab.ab_sync(ctx)                     # reported once, by the call
    again, it2, rr2 = ab.ab_kernel_solve(ctx, X, B, 50.0, 0.25, "fp32", 1e-4, 1000)
    assert it2 == it and rr2 == rr and torch.equal(again, W)
    # a block past the grid is none
    ab.ab_testing_solve_timeout(ctx, 100000, 2_000_000_000)
    again, it2, _ = ab.ab_kernel_solve(ctx, X, B, 50.0, 0.25, "fp32", 1e-4, 1000)
    assert it2 == it and torch.equal(again, W)
    ab.ab_sync(ctx)
    ctx.close()
