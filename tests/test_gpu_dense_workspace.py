"""Memory of the dense entry points: a captured call keeps no pointer that a
later call gives back, a captured call does what an eager one does, calls on
two streams share nothing, and a destroyed context leaves nothing behind
(GPU, C ABI).  Every comparison is bit for bit: the same kernels on the same
inputs."""
import pytest
import torch

pytestmark = pytest.mark.gpu
S = 200.0


@pytest.fixture(scope="module")
def ab():
    import paper_1704_08907_gb300 as ab
    return ab


def _inputs(m, n, nrhs, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = dict(generator=g, device="cuda")
    X, Y = torch.rand((m, 4), **f), torch.rand((n, 4), **f)
    return X, Y, torch.randn((n, nrhs), **f), torch.randn((m, nrhs), **f)


def _outputs(X, Y, W):
    return (torch.zeros_like(W), torch.zeros_like(X), torch.zeros_like(Y),
            torch.zeros((), dtype=torch.float64, device=X.device))


@pytest.mark.parametrize("prec,nrhs", [("bf16x3", 64), ("tf32x3", 64), ("fp32", 64), ("fp32", 3)])
def test_graph_outlives_larger_calls(ab, cuda, prec, nrhs):
    ctx = ab.Context(0)
    X, Y, W, G = _inputs(700, 5000, nrhs, 1)
    out = ab.ab_kernel_matvec(ctx, X, Y, W, S, prec)
    grads = _outputs(X, Y, W)
    ab.ab_kernel_matvec_bwd(ctx, X, Y, W, S, prec, G, *grads)
    ab.ab_sync(ctx)
    got, got_grads = torch.zeros_like(out), _outputs(X, Y, W)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ab.ab_kernel_matvec(ctx, X, Y, W, S, prec, out=got)
        ab.ab_kernel_matvec_bwd(ctx, X, Y, W, S, prec, G, *got_grads)
    # larger eager calls of every precision, then memory for others to write
    big = _inputs(9000, 30000, 64, 2)
    for p in ("fp32", "bf16x3", "tf32x3"):
        ab.ab_kernel_matvec(ctx, *big[:3], S, p)
        ab.ab_kernel_matvec_bwd(ctx, *big[:3], S, p, big[3], *_outputs(*big[:3]))
    ab.ab_sync(ctx)
    junk = [torch.full((1 << 24,), float("nan"), device=cuda) for _ in range(8)]
    for _ in range(2):
        got.zero_()
        for t in got_grads:
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(got, out)
        assert all(torch.equal(a, b) for a, b in zip(got_grads, grads))
    assert all(torch.isnan(j).all() for j in junk)
    # a replay among eager calls
    g.replay()
    again = ab.ab_kernel_matvec(ctx, X, Y, W, S, prec)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(again, out) and torch.equal(got, out)
    ab.ab_sync(ctx)
    ctx.close()


@pytest.mark.parametrize("prec,nrhs", [("fp32", 1), ("fp32", 16), ("bf16x3", 64)])
def test_two_streams(ab, cuda, prec, nrhs):
    ctx = ab.Context(0)
    sets = [_inputs(900, 20000, nrhs, 3), _inputs(1100, 17000, nrhs, 4)]
    want = [ab.ab_kernel_matvec(ctx, *s[:3], S, prec) for s in sets]
    gwant = []
    for s in sets:
        gwant.append(_outputs(*s[:3]))
        ab.ab_kernel_matvec_bwd(ctx, *s[:3], S, prec, s[3], *gwant[-1])
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    got, ggot = [], []
    for k in range(20):
        with torch.cuda.stream(streams[k % 2]):
            s = sets[k % 2]
            got.append(ab.ab_kernel_matvec(ctx, *s[:3], S, prec))
            ggot.append(_outputs(*s[:3]))
            ab.ab_kernel_matvec_bwd(ctx, *s[:3], S, prec, s[3], *ggot[-1])
    torch.cuda.synchronize()
    for k in range(20):
        assert torch.equal(got[k], want[k % 2])
        assert all(torch.equal(a, b) for a, b in zip(ggot[k], gwant[k % 2]))
    ctx.close()


def test_memory_is_given_back(ab, cuda):
    big = _inputs(30000, 60000, 64, 5)
    outs = _outputs(*big[:3])
    res = torch.empty_like(big[3])
    torch.cuda.synchronize()

    def used():
        ctx = ab.Context(0)
        ab.ab_kernel_matvec(ctx, *big[:3], S, "fp32", out=res)
        ab.ab_kernel_matvec_bwd(ctx, *big[:3], S, "fp32", big[3], *outs)
        ab.ab_kernel_matvec(ctx, *big[:3], S, "tf32x3", out=res)
        ab.ab_sync(ctx)
        torch.cuda.synchronize()
        held = torch.cuda.mem_get_info()[0]
        ctx.close()
        torch.cuda.synchronize()
        return held, torch.cuda.mem_get_info()[0]

    used()                                  # modules loaded, default pool warm
    before = torch.cuda.mem_get_info()[0]
    held, after = used()
    assert before - held <= 256 << 20       # the 138 MB of partial sums, a quarter more, the cell list's own
    assert before - after <= 32 << 20


def test_destroyed_while_the_first_stream_runs(ab, cuda):
    """The buffer belongs to the stream of the first dense call; the context is
    destroyed on another one while that stream is still at work."""
    m, n = 4000, 60000
    X, Y, W, _ = _inputs(m, n, 64, 6)
    ctx = ab.Context(0)
    want = ab.ab_kernel_matvec(ctx, X, Y, W, S, "fp32")
    ctx.close()
    got = [torch.zeros_like(want) for _ in range(20)]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx = ab.Context(0)
    with torch.cuda.stream(side):
        for g in got:
            ab.ab_kernel_matvec(ctx, X, Y, W, S, "fp32", out=g)
    ab.ab_kernel_matvec(ctx, X[:10], Y[:10], W[:10], S, "fp32")
    ctx.close()
    other = ab.Context(0)
    last = ab.ab_kernel_matvec(other, X, Y, W, S, "fp32")
    torch.cuda.synchronize()
    assert torch.equal(last, want) and all(torch.equal(g, want) for g in got)
    other.close()
