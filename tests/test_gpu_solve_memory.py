"""Device memory that a context holds after a one-launch solve, which works on
a slab of 4 n^2 bytes: at most 256 MB stay (n = 8,000 and below), the slab of a
larger system goes back, and so does everything with the context (GPU, C ABI).
The other 96 MB are the margin for the allocator's granularity and modules."""
import numpy as np
import pytest
import torch

import synth
from _helpers import dev

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.mark.parametrize("n,most", [(4096, 64 * 5 // 4 + 96), (7900, 256 + 96), (9700, 96)])
def test_slab_is_bounded(cuda, n, most):
    import paper_1704_08907_gb300 as ab
    X = dev(synth.uniform_positions(n, 3, 900 + n))
    B = dev(np.random.default_rng(901).standard_normal((n, 1)).astype(np.float32))
    W = torch.empty_like(B)
    first = None
    for _ in range(2):                   # the first loads the modules
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ctx = ab.Context(0)
        _, it, rr = ab.ab_kernel_solve(ctx, X, B, 200.0, 0.5, "fp32", 1e-4, 1000, W=W)
        assert it > 0 and rr <= 1e-4
        first = W.clone() if first is None else first
        ab.ab_kernel_solve(ctx, X, B, 200.0, 0.5, "fp32", 1e-4, 1000, W=W)
        assert torch.equal(W, first)
        ab.ab_sync(ctx)
        torch.cuda.synchronize()
        held = before - torch.cuda.mem_get_info()[0]
        ctx.close()
        torch.cuda.synchronize()
        left = before - torch.cuda.mem_get_info()[0]
    assert held <= most * MB
    assert left <= 32 * MB
