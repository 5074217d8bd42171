"""Tensor-core gradients of a whole number of waves of row blocks: their FP32
sums over the points run over two ranges like those of fewer rows, so the first
half of the rows gives the same bits whether the other half is there or not
(GPU, C ABI).  76 and 152 row blocks: half a wave and one on 152 SMs."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["bf16x3", "tf32x3", "bf16"])
@pytest.mark.parametrize("n", [9000, 30000])
def test_rows_do_not_depend_on_the_wave(cuda, prec, n):
    import paper_1704_08907_gb300 as ab
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("row blocks chosen for 152 SMs")
    g = torch.Generator(device="cuda").manual_seed(n)
    f = dict(generator=g, device="cuda")
    m = 152 * 128
    X, Y = torch.rand((m, 4), **f), torch.rand((n, 4), **f)
    W, G = torch.rand((n, 64), **f), torch.rand((m, 64), **f)
    ctx = ab.Context(0)
    dX, half = torch.empty_like(X), torch.empty_like(X[:m // 2])
    ab.ab_kernel_matvec_bwd(ctx, X, Y, W, 50.0, prec, G, None, dX)
    ab.ab_kernel_matvec_bwd(ctx, X[:m // 2], Y, W, 50.0, prec, G[:m // 2], None, half)
    assert torch.equal(dX[:m // 2], half)
    # the same for the points' gradient, with the roles swapped
    dY, half = torch.empty_like(X), torch.empty_like(X[:m // 2])
    ab.ab_kernel_matvec_bwd(ctx, Y, X, G, 50.0, prec, W, None, None, dY)
    ab.ab_kernel_matvec_bwd(ctx, Y, X[:m // 2], G[:m // 2], 50.0, prec, W, None, None, half)
    assert torch.equal(dY[:m // 2], half)
    ab.ab_sync(ctx)
    ctx.close()
