"""Totals over per-block FP64 partials at the sizes where their reduction goes
from one block to a cluster of eight (more than 1024 partials) and where the
eight shares are uneven or partly empty: the total energy against the FP64 sum
of the per-particle energies the same call returned (GPU, C ABI).

Tolerance: both sides add the same FP32 values in FP64, so they differ by the
roundings of the additions alone: at most one a particle along the longest
chain (well under 4,096 of them), each half an ulp of a partial sum no larger
than sum |E|: 4096 * 2^-53 < 5e-13 of sum |E|.
"""
import pytest
import torch

import synth
from _helpers import dev

pytestmark = pytest.mark.gpu


# 128 particles a partial at these densities: 1024, 1025, 1032 and 8191 partials
@pytest.mark.parametrize("n", [131072, 131073, 132096, 1048449])
def test_total_energy_is_the_sum(cuda, n):
    import paper_1704_08907_gb300 as ab
    r = float((8.0 * 0.75 / (3.14159265 * n)) ** (1 / 3))
    pos = dev(synth.uniform_positions(n, 3, 4 + n))
    ctx = ab.Context(0)
    ab.ab_build(ctx, ab.Domain(3, (1, 1, 1), r), pos)
    prm = ab.OpParams(eps=1.0, sigma=0.02 * r)
    E, _, total = ab.ab_pair_energy_grad(ctx, "lj", prm)
    ab.ab_sync(ctx)
    e = E.double()
    assert torch.isfinite(e).all()
    assert abs(float(total) - float(e.sum())) <= 5e-13 * float(e.abs().sum())
    again = [float(ab.ab_pair_energy_grad(ctx, "lj", prm)[2]) for _ in range(3)]
    assert again == [float(total)] * 3
    ctx.close()
