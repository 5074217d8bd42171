"""FP32 dense operator with rows of whole float4s, which are moved 16 bytes at a
time when they are aligned (8 columns and more), against the same call on
buffers aligned to 4 bytes only: the same bits, since only the copies differ
(GPU, C ABI).  Remainders of columns, stages and row blocks, split and not."""
import pytest
import torch

import synth
from _helpers import dev
from test_gpu_dense import _dev4

pytestmark = pytest.mark.gpu


def _shift(t):
    """The same values, 4 bytes past a 16-byte boundary."""
    return torch.cat([torch.zeros(1, device=t.device), t.reshape(-1)])[1:].view(t.shape)


@pytest.mark.parametrize("m,n,nrhs", [(1, 130, 8), (513, 4001, 8), (300, 65, 12), (700, 3000, 16), (257, 129, 20),
                                      (511, 1000, 32), (100, 63, 40), (600, 700, 64)])
def test_aligned_rows(cuda, m, n, nrhs):
    import paper_1704_08907_gb300 as ab

    d = synth.c4(m=m, n=n, nrhs=nrhs, seed_offset=3000 + m + n)
    ctx = ab.Context(0)
    X, Y = _dev4(d.X), _dev4(d.Y)
    got = []
    for move in (lambda t: t, _shift):
        W, G = move(dev(d.W)), move(dev(d.G))
        assert W.data_ptr() % 16 == (4 if got else 0)
        out, dW = move(torch.zeros((m, nrhs), device=cuda)), move(torch.zeros((n, nrhs), device=cuda))
        dX, dY = torch.empty_like(X), torch.empty_like(Y)
        ds = torch.empty((), dtype=torch.float64, device=cuda)
        ab.ab_kernel_matvec(ctx, X, Y, W, d.s, "fp32", out=out)
        ab.ab_kernel_matvec_bwd(ctx, X, Y, W, d.s, "fp32", G, dW, dX, dY, ds)
        ab.ab_sync(ctx)
        got.append((out, dW, dX, dY, ds))
    for a, b in zip(*got):
        assert torch.equal(a, b)
    ctx.close()
