"""Pair sums over the sizes at which the number of lanes that share a
particle's walk changes (1, 2, 4, 8, 32), with particle counts that leave a
remainder in the last warp and block: values and adjoints against the FP64
oracle (the metric and the 1e-5 of tests/test_gpu_pairsum.py: sharing only
regroups the sum), and the one-walk calls against the separate ones bit for
bit (GPU, C ABI)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from _helpers import dev, host, rel_err

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def ab():
    import paper_1704_08907_gb300 as ab
    return ab


# dim, n, mean neighbours, periodic, blobs
CASES = {
    "long_rows_general": (2, 3001, 600.0, (1, 1), 0),
    "long_rows": (2, 20001, 400.0, (1, 0), 0),
    "long_rows_wide": (2, 98305, 300.0, (1, 1), 0),
    "mid_rows_small": (2, 4097, 77.0, (1, 1), 0),
    "small_3d": (3, 5003, 33.6, (1, 0, 1), 0),
    "small_2d": (2, 16383, 9.4, (0, 0), 0),
    "clustered_small": (3, 5120, 20.0, (1, 1, 1), 4),
    "quarter_3d": (3, 40001, 33.6, (1, 1, 1), 0),
    "quarter_2d": (2, 40001, 9.4, (1, 1), 0),
    "half_3d": (3, 131073, 25.0, (1, 1, 0), 0),
    "full_3d": (3, 262145, 20.0, (1, 1, 1), 0),
    "tiny": (3, 3, 0.1, (1, 1, 1), 0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_values_and_adjoints(ab, cuda, name):
    dim, n, nb, periodic, blobs = CASES[name]
    if blobs:
        pos = synth.blob_positions(n, blobs, 0.01, 70)
        r = 0.004
    else:
        pos = synth.uniform_positions(n, dim, 71 + n)
        r = np.sqrt(nb / (np.pi * n)) if dim == 2 else (nb * 0.75 / (np.pi * n)) ** (1 / 3)
    r = float(np.float32(r))
    ctx = ab.Context(0)
    ab.ab_build(ctx, ab.Domain(dim, periodic, r), dev(pos))
    box = oracle.Box(dim, periodic, radius=r)
    off, idx = oracle.CellList(box, pos).neighbours(None)
    w, g = synth.weights(n, 72), synth.weights(n, 73, "normal")

    cnt = host(ab.ab_pair_sum(ctx, "count", ab.OpParams()))
    assert np.array_equal(cnt, np.diff(off).astype(np.float32))
    s = 9.0 / r ** 2
    y = ab.ab_pair_sum(ctx, "gauss", ab.OpParams(s=s), w=dev(w))
    p = {"s": s}
    assert rel_err(host(y), oracle.pair_values("gauss", box, pos, off, idx, w=w, params=p)[:, 0],
                   oracle.abs_terms("gauss", box, pos, off, idx, w=w, params=p)[:, 0]) <= TOL
    for op, prm, p in (("expf", ab.OpParams(c=0.5), {"c": 0.5}), ("soft", ab.OpParams(k=3.0), {"k": 3.0})):
        f = host(ab.ab_pair_sum(ctx, op, prm))
        assert rel_err(f[:, :dim], oracle.pair_values(op, box, pos, off, idx, params=p)[:, :dim],
                       oracle.abs_terms(op, box, pos, off, idx, params=p)[:, :dim]) <= TOL
        assert np.all(f[:, dim:] == 0)

    # Gaussian adjoint, and the values in the same walk
    f32, f64 = dict(dtype=torch.float32, device=cuda), dict(dtype=torch.float64, device=cuda)
    gp, gw, gs = torch.empty((n, 4), **f32), torch.empty(n, **f32), torch.empty((), **f64)
    ab.ab_pair_sum_bwd(ctx, "gauss", ab.OpParams(s=s), dev(w), dev(g), gp, gw, gs)
    ref, rw, rs = oracle.pair_grads("gauss", box, pos, off, idx, g, w=w, params={"s": s})
    den, dw, ds = oracle.abs_grad_terms("gauss", box, pos, off, idx, g, w=w, params={"s": s})
    assert rel_err(host(gp)[:, :dim], ref[:, :dim], den[:, :dim]) <= TOL
    assert rel_err(host(gw), rw, dw) <= TOL
    assert abs(float(gs) - rs.sum()) <= TOL * max(ds.sum(), 1e-30)
    y2, gp2, gw2, gs2 = torch.empty(n, **f32), torch.empty_like(gp), torch.empty_like(gw), torch.empty((), **f64)
    ab.ab_pair_sum_value_grad(ctx, "gauss", ab.OpParams(s=s), dev(w), dev(g), y2, None, gp2, gw2, gs2)
    for a, b in ((y, y2), (gp, gp2), (gw, gw2), (gs, gs2)):
        assert torch.equal(a, b)

    # LJ: the fused energy and gradient are the separate calls' bits
    lj = ab.OpParams(eps=1.0, sigma=0.3 * r)
    e0, e1 = torch.empty((), **f64), torch.empty((), **f64)
    E0 = ab.ab_pair_sum(ctx, "lj", lj, energy=e0)
    F0 = torch.empty((n, 4), **f32)
    ab.ab_pair_sum_bwd(ctx, "lj", lj, None, torch.ones(n, **f32), F0)
    E1, F1, _ = ab.ab_pair_energy_grad(ctx, "lj", lj, energy=e1)
    assert torch.equal(E0, E1) and torch.equal(F0, F1) and torch.equal(e0, e1)
    p = {"eps": 1.0, "sigma": 0.3 * r}
    assert rel_err(host(E0), oracle.pair_values("lj", box, pos, off, idx, params=p)[:, 0],
                   oracle.abs_terms("lj", box, pos, off, idx, params=p)[:, 0]) <= TOL
    ab.ab_sync(ctx)
    ctx.close()
