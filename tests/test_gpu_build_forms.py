"""Every form of the build at the edges of its range, with the form that ran
checked, against the kernel sequence bit for bit: one block up to 6,144
particles (and up to 8,192 where the cluster is not taken), a cluster of 16
blocks from 6,145 to 16,384 and up to 32 particles a cell, tables around the
shared memory of either, half of the particles in a few cells of a table that
keeps the cluster (its loads of four slots), packed positions (GPU)."""
import numpy as np
import pytest

import synth
from _helpers import dev
from test_gpu_build_small import _list

pytestmark = pytest.mark.gpu
BLOCK, CLUSTER, COOP = "BLOCK", "CLUSTER", "COOP"

# dim, n, cells per axis (radius 1 / (cells + 0.5), not periodic), crowded
CASES = [
    (2, 4097, 20, 0, BLOCK), (3, 5001, 9, 0, BLOCK), (2, 6144, 20, 0, BLOCK), (3, 6144, 9, 0, BLOCK),
    (2, 6000, 25, 1, BLOCK), (2, 6145, 20, 0, CLUSTER), (3, 6145, 9, 0, CLUSTER), (2, 8193, 30, 0, CLUSTER),
    (2, 16383, 40, 0, CLUSTER), (3, 16384, 12, 0, CLUSTER), (2, 16384, 40, 0, CLUSTER),
    (2, 16385, 40, 0, COOP), (3, 16385, 12, 0, COOP),
    (2, 12000, 30, 1, CLUSTER), (3, 16000, 10, 1, CLUSTER), (2, 6145, 20, 1, CLUSTER), (2, 16384, 40, 1, CLUSTER),
    # cells that the blocks of the cluster share unevenly
    (2, 7001, 8, 0, CLUSTER), (3, 7003, 6, 0, CLUSTER),
]


@pytest.mark.parametrize("dim,n,cells,crowded,form", CASES)
@pytest.mark.parametrize("packed", [False, True])
def test_form_and_list(cuda, dim, n, cells, crowded, form, packed):
    import paper_1704_08907_gb300 as ab
    pos = synth.uniform_positions(n, dim, 950 + n + cells)
    if crowded:      # half of the points around four places, the rest spread
        centre = np.float32([0.13, 0.37, 0.61, 0.88])[np.arange(n // 2) % 4, None]
        pos[: n // 2, :dim] = centre + pos[: n // 2, :dim] * np.float32(1e-3)
    dom = ab.Domain(dim, (0, 0, 0)[:dim], 1.0 / (cells + 0.5))
    p = dev(pos[:, :dim].copy()) if packed else dev(pos)
    ctx = ab.Context(0)
    ab.ab_testing_cell_table(ctx, 1)
    a = _list(ab, ctx, dom, p, ab.BUILD_AUTO)
    assert ab.ab_testing_build_form(ctx) == getattr(ab, "FORM_" + form)
    b = _list(ab, ctx, dom, p, ab.BUILD_SEQUENCE)
    assert ab.ab_testing_build_form(ctx) == ab.FORM_SEQUENCE
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    if crowded:
        assert np.diff(a[1].astype(np.int64)).max() >= 400
    ctx.close()


# 2 x rows cells, periodic: 32 particles a cell is the cluster's limit, past it
# one block or the cooperative launch, which also takes over from one block
# above 2,048 particles at n^2 = 240,000 cells; 195 table entries, 13 a block,
# leave the cluster's last block without any
@pytest.mark.parametrize("rows,n,form", [(97, 6208, CLUSTER), (97, 6209, BLOCK), (128, 8192, CLUSTER),
                                         (1, 2048, BLOCK), (4, 2049, COOP), (30, 3790, BLOCK),
                                         (30, 3796, COOP), (127, 8192, COOP), (200, 12800, CLUSTER), (200, 12801, COOP)])
def test_particles_a_cell(cuda, rows, n, form):
    import paper_1704_08907_gb300 as ab
    r = 0.125
    hi = (2.5 * r, (rows + 0.5) * r)
    pos = synth.uniform_positions(n, 2, 970 + n)
    pos[:, :2] *= np.float32(0.999) * np.float32(hi)
    dom = ab.Domain(2, (1, 1), r, hi=hi)
    ctx = ab.Context(0)
    ab.ab_testing_cell_table(ctx, 1)
    a = _list(ab, ctx, dom, dev(pos), ab.BUILD_AUTO)
    assert ab.ab_cell_shape(ctx)[1] == 2 * rows
    ab.ab_testing_build_path(ctx, ab.BUILD_AUTO)
    ab.ab_build(ctx, dom, dev(pos))
    assert ab.ab_testing_build_form(ctx) == getattr(ab, "FORM_" + form)
    b = _list(ab, ctx, dom, dev(pos), ab.BUILD_SEQUENCE)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    ctx.close()
