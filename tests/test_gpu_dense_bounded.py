"""Partial sums of the FP32 dense walk: what a context holds after a product
and an adjoint of many rows stays within the bound (224 MB and the quarter that
buffers grow by; 64 MB more for the allocator's granularity), and rows and points
on both sides of the bound agree with FP64 (GPU, C ABI; metric and 1e-5 of
tests/test_gpu_dense.py on sampled rows)."""
import pytest
import torch

pytestmark = pytest.mark.gpu
MB = 1 << 20


@pytest.mark.parametrize("m,n,nrhs", [(400000, 20000, 64), (65536, 20000, 64), (300000, 9001, 32)])
def test_held_memory_and_rows(cuda, m, n, nrhs):
    import paper_1704_08907_gb300 as ab
    g = torch.Generator(device="cuda").manual_seed(m)
    f = dict(generator=g, device="cuda")
    X, Y = torch.rand((m, 4), **f), torch.rand((n, 4), **f)
    W, G = torch.randn((n, nrhs), **f), torch.randn((m, nrhs), **f)
    out, dW, dX, dY = torch.empty_like(G), torch.empty_like(W), torch.empty_like(X), torch.empty_like(Y)
    s = 60.0
    for _ in range(2):                    # the first loads the modules
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        ctx = ab.Context(0)
        ab.ab_kernel_matvec(ctx, X, Y, W, s, "fp32", out=out)
        ab.ab_kernel_matvec_bwd(ctx, X, Y, W, s, "fp32", G, dW, dX, dY)
        ab.ab_sync(ctx)
        torch.cuda.synchronize()
        held = before - torch.cuda.mem_get_info()[0]
        ctx.close()
        torch.cuda.synchronize()
    assert held <= (224 * 5 // 4 + 64) * MB

    def check(got, P, Q, V, k):
        idx = torch.randint(0, P.shape[0], (64,), generator=torch.Generator().manual_seed(k)).cuda()
        d2 = ((P[idx, None, :3].double() - Q[None, :, :3].double()) ** 2).sum(-1)
        K = torch.exp(-s * d2)
        assert float(((got[idx].double() - K @ V.double()).abs() / (K @ V.double().abs())).max()) <= 1e-5

    check(out, X, Y, W, 1)
    check(dW, Y, X, G, 2)
