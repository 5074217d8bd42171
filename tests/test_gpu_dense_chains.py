"""FP32 gradients and ds where nothing averages out: all rows at one place, all
points at another, so that every term of a row's sum is the same and each
addition may round the same way (GPU, C ABI).  Row counts that fill the SMs in
whole waves are not split over the points, so a row's sum is one thread's.

Tolerance: the sums run over at most 512 points and then over those sums (256
points at 64 columns), so a sum of n terms meets at most 512 + n / 256 roundings
of 2^-24 (and a few for the ranges, the factor and ds's block); a chain over all
points would meet n, off by 2.9e-4 here.  K, the same for all pairs, adds the 2^-22 of
ex2 and the rounding of its exponent (8 * 2^-24)."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu


# waves of row blocks (256 rows; 4, 3 and 2 a SM) at 1, 16, 32 and 64 columns
@pytest.mark.parametrize("nrhs,per_sm", [(1, 4), (4, 4), (16, 3), (32, 2), (64, 2)])
def test_equal_terms(cuda, nrhs, per_sm):
    import paper_1704_08907_gb300 as ab
    m = 256 * per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    n = 20011
    ctx = ab.Context(0)
    X = torch.zeros((m, 4), device=cuda)
    Y = torch.zeros((n, 4), device=cuda)
    Y[:, 0] = 0.5
    tol = (512 + n / 256 + 16) * 2.0 ** -24 + 2.0 ** -22 + 8 * 2.0 ** -24
    for s, w in ((1.0, 1.0), (1.7, 0.7), (3.1, 0.3), (0.37, 0.9)):
        W = torch.full((n, nrhs), w, device=cuda)
        G = torch.ones((m, nrhs), device=cuda)
        dX, dY = torch.empty_like(X), torch.empty_like(Y)
        ds = torch.empty((), dtype=torch.float64, device=cuda)
        sf, wf = float(torch.tensor(s, dtype=torch.float32)), float(W[0, 0])
        a = nrhs * wf * math.exp(-sf * 0.25)          # (G_i . W_j) K_ij
        ab.ab_kernel_matvec_bwd(ctx, X, Y, W, s, "fp32", G, None, dX, dY, ds)
        ab.ab_sync(ctx)
        for got, count, sign in ((dX, n, 1.0), (dY, m, -1.0)):
            want = sign * 2.0 * sf * a * 0.5 * count
            bound = tol if count == n else tol + (m - n) / 256 * 2.0 ** -24
            assert float((got[:, 0].double() / want - 1).abs().max()) <= bound
            assert torch.all(got[:, 1:] == 0)
        assert abs(float(ds) / (-a * 0.25 * m * n) - 1) <= tol
    # one walk for dW and dY
    if nrhs <= 32:
        dW, dY = torch.empty((m, nrhs), device=cuda), torch.empty_like(X)
        ab.ab_kernel_matvec_bwd(ctx, Y, X, torch.ones((m, nrhs), device=cuda), s, "fp32", W, dW, None, dY)
        want = 2.0 * sf * a * 0.5 * n
        assert float((dY[:, 0].double() / want - 1).abs().max()) <= tol
    ab.ab_sync(ctx)
    ctx.close()
