"""The build over a thread-block cluster against the kernel sequence, bit for
bit, at the edges of its range: one past the one-block build, one, two and four
particles a thread with remainders, the first count beyond it, cell tables
that leave blocks of the cluster without cells, crowded cells, packed
positions; and replayed from a graph (GPU)."""
import numpy as np
import pytest
import torch

import synth
from _helpers import dev, host
from test_gpu_build_small import _list

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,r,crowded", [
    (2, 8193, 0.01, 0), (3, 8193, 0.45, 0), (2, 16384, 0.006, 0), (3, 16385, 0.05, 0), (2, 20000, 0.2, 0),
    (3, 32767, 0.03, 0), (2, 32768, 0.004, 0), (2, 32769, 0.004, 0), (3, 20000, 0.1, 1), (2, 9001, 0.3, 1),
    (2, 65536, 0.003, 0), (3, 65537, 0.03, 0)])
@pytest.mark.parametrize("packed", [False, True])
def test_equals_kernel_sequence(cuda, dim, n, r, crowded, packed):
    import paper_1704_08907_gb300 as ab

    pos = synth.uniform_positions(n, dim, 900 + n)
    if crowded:      # half of the points in one cell, the rest spread
        pos[: n // 2, :dim] = np.float32(0.5) + pos[: n // 2, :dim] * np.float32(1e-3)
    dom = ab.Domain(dim, (1, 0, 1)[:dim], r)
    p = dev(pos[:, :dim].copy()) if packed else dev(pos)
    ctx = ab.Context(0)
    ab.ab_testing_cell_table(ctx, 1)
    a = _list(ab, ctx, dom, p, ab.BUILD_AUTO)
    b = _list(ab, ctx, dom, p, ab.BUILD_SEQUENCE)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    ctx.close()


def test_replayed(cuda):
    import paper_1704_08907_gb300 as ab

    n = 12345
    ctx, dom = ab.Context(0), ab.Domain(2, (1, 1), 0.01)
    p, q = (dev(synth.uniform_positions(n, 2, k)) for k in (7, 8))
    ref = _list(ab, ctx, dom, q, ab.BUILD_SEQUENCE)
    ab.ab_testing_build_path(ctx, ab.BUILD_AUTO)
    out = torch.empty(n, dtype=torch.float32, device=cuda)
    ab.ab_build(ctx, dom, p)
    ab.ab_pair_sum(ctx, "count", ab.OpParams(), out=out)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ab.ab_build(ctx, dom, p)
        ab.ab_pair_sum(ctx, "count", ab.OpParams(), out=out)
    p.copy_(q)
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(host(out), ref[2])
    ctx.close()
