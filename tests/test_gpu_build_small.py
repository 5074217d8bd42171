"""The one-block build against the kernel sequence, bit for bit, at the edges
of its range: particle counts around a block and its per-thread counts (1024,
4096, 8192, and one more, where the cooperative form takes over), cell tables
around its shared memory, crowded and empty cells, packed positions (GPU)."""
import numpy as np
import pytest
import torch

import synth
from _helpers import dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ab():
    import paper_1704_08907_gb300 as ab
    return ab


def _list(ab, ctx, dom, p, path):
    ab.ab_testing_build_path(ctx, path)
    ab.ab_build(ctx, dom, p)
    perm, start = ab.ab_cell_export(ctx)
    c = ab.ab_pair_sum(ctx, "count", ab.OpParams())
    ab.ab_sync(ctx)
    return host(perm), host(start), host(c)


@pytest.mark.parametrize("dim,n,r,crowded", [
    (2, 1, 0.1, 0), (2, 33, 0.3, 0), (3, 1023, 0.1, 0), (2, 1025, 0.02, 0), (3, 4096, 0.05, 0),
    (2, 4097, 0.01, 0), (3, 8191, 0.04, 0), (2, 8192, 0.0062, 0), (2, 8193, 0.0062, 0),
    (2, 8000, 0.0112, 0), (2, 8000, 0.0118, 0), (2, 3000, 0.05, 1), (3, 5001, 0.3, 1), (3, 2, 0.49, 0)])
@pytest.mark.parametrize("packed", [False, True])
def test_equals_kernel_sequence(ab, cuda, dim, n, r, crowded, packed):
    pos = synth.uniform_positions(n, dim, 800 + n)
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


def test_cooperative_builds_follow_one_another(ab, cuda):
    """The barrier words are cleared by each launch for the next: builds of
    different sizes, eager and replayed from a graph, after one that timed
    out."""
    ctx = ab.Context(0)
    ab.ab_testing_build_path(ctx, ab.BUILD_COOP)
    big, small = synth.uniform_positions(300000, 2, 5), synth.uniform_positions(9000, 2, 6)
    dom = ab.Domain(2, (1, 1), 0.01)
    db, ds = dev(big), dev(small)
    ref = {}
    for name, p in (("big", db), ("small", ds)):
        ref[name] = _list(ab, ctx, dom, p, ab.BUILD_SEQUENCE)
    for name, p in (("big", db), ("small", ds), ("big", db)):
        for x, y in zip(_list(ab, ctx, dom, p, ab.BUILD_COOP), ref[name]):
            assert np.array_equal(x, y)
    out = torch.empty(300000, dtype=torch.float32, device=cuda)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ab.ab_build(ctx, dom, db)
        ab.ab_pair_sum(ctx, "count", ab.OpParams(), out=out)
    ab.ab_testing_build_timeout(ctx, 0, 5_000_000)
    ab.ab_build(ctx, dom, db)
    with pytest.raises(ab.AbError) as e:
        ab.ab_sync(ctx)
    assert e.value.status == 6
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(host(out), ref["big"][2])
    ab.ab_sync(ctx)
    ctx.close()
