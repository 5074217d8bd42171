"""FP32 dense operator and adjoint over the sizes at which its walk changes
(GPU, C ABI): each compiled column count and the next odd one, row blocks of
256 and 512 with remainders, other points split over blocks or not, stages of
64 and 128 points with remainders.

Error metrics as tests/test_gpu_dense.py, all <= 1e-5: a sum of N FP32 terms
with relative rounding 2^-24 each stays below N 2^-24 of the terms' magnitudes
in the worst case and below sqrt(N) 2^-24 in practice (2e-6 at the largest N
here), and each term carries about 4 roundings and ex2's 2^-22."""
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


SHAPES = [(1, 1, 1), (1, 5000, 1), (5000, 1, 2), (511, 513, 1), (513, 127, 2), (257, 129, 3),
          (255, 65, 4), (512, 128, 5), (640, 1000, 8), (100, 3001, 9), (3001, 100, 16),
          (130, 700, 17), (700, 130, 32), (259, 300, 33), (300, 259, 64), (1500, 1400, 1)]


@pytest.mark.parametrize("m,n,nrhs", SHAPES)
def test_forward_and_adjoint(ab, cuda, m, n, nrhs):
    d = synth.c4(m=m, n=n, nrhs=nrhs, seed_offset=1000 + m + n)
    ctx = ab.Context(0)
    X, Y = _dev4(d.X), _dev4(d.Y)
    # weights 4-byte aligned only
    W = torch.cat([torch.zeros(1, device=cuda), dev(d.W).reshape(-1)])[1:].view(n, nrhs)
    G = torch.cat([torch.zeros(1, device=cuda), dev(d.G).reshape(-1)])[1:].view(m, nrhs)
    out = ab.ab_kernel_matvec(ctx, X, Y, W, d.s, "fp32")
    ref, den = dense.matvec(d.X, d.Y, d.W, d.s), dense.matvec_abs(d.X, d.Y, d.W, d.s)
    assert np.max(np.abs(host(out) - ref) / den) <= 1e-5
    dW, dX, dY = torch.empty_like(W), torch.empty_like(X), torch.empty_like(Y)
    ds = torch.empty((), dtype=torch.float64, device=cuda)
    ab.ab_kernel_matvec_bwd(ctx, X, Y, W, d.s, "fp32", G, dW, dX, dY, ds)
    ab.ab_sync(ctx)
    rW, aW = dense.grad_W(d.X, d.Y, d.G, d.s), dense.grad_W(d.X, d.Y, np.abs(d.G), d.s)
    assert np.max(np.abs(host(dW) - rW) / aW) <= 1e-5
    _check_dxdy(d, dX, dY, 1e-5)
    assert np.all(host(dX)[:, 3] == 0) and np.all(host(dY)[:, 3] == 0)
    rs, As = dense.grad_s(d.X, d.Y, d.W, d.G, d.s), dense.grad_s_abs(d.X, d.Y, d.W, d.G, d.s)
    assert abs(float(ds) - rs) <= 1e-5 * As
    # each output alone, and the same call again, give the same bits (one
    # walk serves dW and dY together when both are wanted)
    for k, want in enumerate((dW, dX, dY)):
        one = torch.empty_like(want)
        ab.ab_kernel_matvec_bwd(ctx, X, Y, W, d.s, "fp32", G, *[one if q == k else None for q in range(3)])
        if k == 1:
            assert torch.equal(one, want)
        else:
            assert torch.allclose(one, want, rtol=1e-4, atol=1e-5 * float(want.abs().max()))
    assert torch.equal(ab.ab_kernel_matvec(ctx, X, Y, W, d.s, "fp32"), out)
    ctx.close()


def test_captured_without_warm_up(ab, cuda):
    """A graph of a context's first FP32 product: no workspace, same sums."""
    d = synth.c4(m=300, n=4000, nrhs=3, seed_offset=4)
    ctx = ab.Context(0)
    X, Y, W = _dev4(d.X), _dev4(d.Y), dev(d.W)
    out = torch.zeros((300, 3), device=cuda)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ab.ab_kernel_matvec(ctx, X, Y, W, d.s, "fp32", out=out)
    g.replay()
    torch.cuda.synchronize()
    ref, den = dense.matvec(d.X, d.Y, d.W, d.s), dense.matvec_abs(d.X, d.Y, d.W, d.s)
    assert np.max(np.abs(host(out) - ref) / den) <= 1e-5
    ab.ab_kernel_matvec(ctx, X, Y, W, d.s, "fp32", out=out)
    assert np.max(np.abs(host(out) - ref) / den) <= 1e-5
    ctx.close()
