"""A captured pair sum keeps its block partials through eager calls with no
more particles but more lanes a particle, hence more blocks (GPU, C ABI): the
replay gives the eager total bit for bit."""
import pytest
import torch

import synth
from _helpers import dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,small", [(300000, 98304), (1500, 1500), (5000, 4096)])
def test_total_survives_calls_with_more_blocks(cuda, n, small):
    import paper_1704_08907_gb300 as ab
    ctx = ab.Context(0)
    pos = dev(synth.uniform_positions(n, 2, 21))
    r = (4.0 / (3.14159265 * n)) ** 0.5           # short rows: few lanes a particle
    dom, prm = ab.Domain(2, (1, 1), r), ab.OpParams(eps=1.0, sigma=0.05 * r)
    E = torch.empty(n, device=cuda)
    total, got = (torch.zeros((), dtype=torch.float64, device=cuda) for _ in range(2))
    ab.ab_build(ctx, dom, pos)
    ab.ab_pair_sum(ctx, "lj", prm, out=E, energy=total)
    ab.ab_sync(ctx)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ab.ab_build(ctx, dom, pos)
        ab.ab_pair_sum(ctx, "lj", prm, out=E, energy=got)
    # long rows: 32 lanes a particle (no more cells than the captured build's)
    wide = min((1200.0 / (3.14159265 * small)) ** 0.5, 0.45)
    ab.ab_build(ctx, ab.Domain(2, (1, 1), wide), pos[:small].contiguous())
    E2 = torch.empty(small, device=cuda)
    total2 = torch.zeros((), dtype=torch.float64, device=cuda)
    ab.ab_pair_sum(ctx, "lj", ab.OpParams(eps=1.0, sigma=1e-4 * wide), out=E2, energy=total2)
    ab.ab_sync(ctx)
    junk = [torch.full((k,), float("nan"), device=cuda) for k in (1 << 10, 1 << 15, 1 << 20)]
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(got, total) and torch.isfinite(got)
    assert all(torch.isnan(j).all() for j in junk)
    ab.ab_sync(ctx)
    ctx.close()
