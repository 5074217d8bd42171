"""Tensor-core dense operator over the sizes at which its rows' sums are split
differently (one range of points, two summed in place, several combined), with
remainders in rows, tiles and ranges: forward and adjoint against the FP64
oracle (the metrics and the 1e-4 of tests/test_gpu_dense.py; splitting only
regroups FP32 sums), each output alone against the full call, and a graph of a
call against the eager one (GPU, C ABI)."""
import numpy as np
import pytest
import torch

import synth
from _helpers import dev, host
from oracle import dense
from test_gpu_dense import _check_dxdy, _dev4

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ab():
    import paper_1704_08907_gb300 as ab
    return ab


@pytest.mark.parametrize("prec", ["bf16x3", "tf32x3"])
@pytest.mark.parametrize("m,n", [(1, 1), (129, 255), (100, 6001), (6001, 100), (2000, 4100), (4097, 300)])
def test_forward_and_adjoint(ab, cuda, prec, m, n):
    d = synth.c4(m=m, n=n, nrhs=64, seed_offset=2000 + m + n)
    ctx = ab.Context(0)
    X, Y, W, G = _dev4(d.X), _dev4(d.Y), dev(d.W), dev(d.G)
    out = ab.ab_kernel_matvec(ctx, X, Y, W, d.s, prec)
    ref, den = dense.matvec(d.X, d.Y, d.W, d.s), dense.matvec_abs(d.X, d.Y, d.W, d.s)
    assert np.max(np.abs(host(out) - ref) / den) <= 1e-4
    dW, dX, dY = torch.empty_like(W), torch.empty_like(X), torch.empty_like(Y)
    ds = torch.empty((), dtype=torch.float64, device=cuda)
    ab.ab_kernel_matvec_bwd(ctx, X, Y, W, d.s, prec, G, dW, dX, dY, ds)
    ab.ab_sync(ctx)
    rW, aW = dense.grad_W(d.X, d.Y, d.G, d.s), dense.grad_W(d.X, d.Y, np.abs(d.G), d.s)
    assert np.max(np.abs(host(dW) - rW) / aW) <= 1e-4
    _check_dxdy(d, dX, dY, 1e-4)
    rs, As = dense.grad_s(d.X, d.Y, d.W, d.G, d.s), dense.grad_s_abs(d.X, d.Y, d.W, d.G, d.s)
    assert abs(float(ds) - rs) <= 1e-4 * As
    # each output alone: the same bits
    for k, want in enumerate((dW, dX, dY, ds)):
        one = torch.empty_like(want)
        ab.ab_kernel_matvec_bwd(ctx, X, Y, W, d.s, prec, G, *[one if q == k else None for q in range(4)])
        assert torch.equal(one, want)
    g = torch.cuda.CUDAGraph()
    got = torch.zeros_like(out)
    with torch.cuda.graph(g):
        ab.ab_kernel_matvec(ctx, X, Y, W, d.s, prec, out=got)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(got, out)
    ab.ab_sync(ctx)
    ctx.close()


@pytest.mark.parametrize("m,n", [(0, 50), (50, 0)])
def test_empty_sides(ab, cuda, m, n):
    ctx = ab.Context(0)
    f = dict(dtype=torch.float32, device=cuda)
    X, Y = torch.rand((m, 4), **f), torch.rand((n, 4), **f)
    W, G = torch.rand((n, 64), **f), torch.rand((m, 64), **f)
    out = ab.ab_kernel_matvec(ctx, X, Y, W, 50.0, "bf16x3", out=torch.ones((m, 64), **f))
    assert torch.all(out == 0)
    dW, dX, dY = torch.ones_like(W), torch.ones_like(X), torch.ones_like(Y)
    ds = torch.ones((), dtype=torch.float64, device=cuda)
    for prec in ("bf16x3", "fp32"):
        ab.ab_kernel_matvec_bwd(ctx, X, Y, W, 50.0, prec, G, dW, dX, dY, ds)
        for t in (dW, dX, dY, ds):
            assert torch.all(t == 0)
    ab.ab_sync(ctx)
    ctx.close()
