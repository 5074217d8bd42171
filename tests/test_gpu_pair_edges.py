"""Coincident points, particles without neighbours and factors near the ends of
FP32 through the vector sums (GPU, C ABI): what has no term is exactly 0, and a
sum that FP32 can hold comes out as FP64 has it.

Two particles at one place, two at a distance of 0.4 r from each other, one
alone.  A term is a handful of FP32 operations with approximate reciprocals and
exponentials, each within 2^-22: 16 * 2^-22 < 4e-6 of it, and no sum here has
more than two."""
import math

import numpy as np
import pytest
import torch

from _helpers import dev, host

pytestmark = pytest.mark.gpu


def _reference(op, dim, x, r, c, k, m, A):
    n = len(x)
    out = np.zeros((n, 3))
    a = 21.0 / (2.0 * math.pi * r ** 3) if dim == 3 else 7.0 / (math.pi * r ** 2)
    for i in range(n):
        for j in range(n):
            dx = x[j] - x[i]
            d = math.sqrt((dx * dx).sum())
            if i == j or d >= r or d == 0.0:
                continue
            if op == "expf":
                f = -c * math.exp(-d) / d
            elif op == "soft":
                f = -k * (r - d) / d
            else:
                f = -20.0 * a / r ** 2 * (m[j] * (A[i] + A[j])) * (1.0 - d / r) ** 3
            out[i, :dim] += np.where(dx == 0.0, 0.0, f * np.where(dx == 0.0, 1.0, dx))
    return out


CASES = [("expf", 1.0, dict(c=1.0)), ("expf", 1.0, dict(c=3e37)), ("expf", 1.0, dict(c=float("inf"))),
         ("soft", 1.0, dict(k=1.0)), ("soft", 1.0, dict(k=2e19)), ("soft", 1.0, dict(k=1e30)),
         ("soft", 1.0, dict(k=-1e37)), ("soft", 1e12, dict(k=1e20)), ("soft", 1e-6, dict(k=1e30)),
         ("soft", 1.0, dict(k=float("inf"))),
         ("sph_force", 1.0, dict(m=1.0, A=1.0)), ("sph_force", 1e-7, dict(m=1e-20, A=0.1)),
         ("sph_force", 1e3, dict(m=1e35, A=50.0)), ("sph_force", 1e-6, dict(m=1e-30, A=1e-3))]


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("op,r,p", CASES)
def test_no_term_is_zero(cuda, dim, op, r, p):
    import paper_1704_08907_gb300 as ab
    r = float(np.float32(r))
    box = 10.0 * r
    x = np.array([[1.0, 1.0, 1.0], [1.0, 1.0, 1.0], [5.0, 5.0, 5.0], [5.4, 5.0, 5.0], [8.0, 2.0, 3.0]])
    pos = np.zeros((5, 4), np.float32)
    pos[:, :dim] = (x * r)[:, :dim]
    x = pos[:, :dim].astype(np.float64)
    m, A = np.full(5, p.get("m", 1.0), np.float32), np.full(5, p.get("A", 1.0), np.float32)
    ctx = ab.Context(0)
    for periodic in ((0, 0, 0), (1, 1, 1)):
        ab.ab_build(ctx, ab.Domain(dim, periodic, r, hi=(box,) * 3), dev(pos))
        w = dev(np.stack([m, A], 1)) if op == "sph_force" else None
        prm = ab.OpParams(c=p.get("c", 1.0), k=p.get("k", 1.0))
        out = host(ab.ab_pair_sum(ctx, op, prm, w=w))
        ab.ab_sync(ctx)
        for i in (0, 1, 4):
            assert np.all(out[i] == 0.0)
        ref = _reference(op, dim, x, r, p.get("c", 1.0), p.get("k", 1.0), m.astype(float), A.astype(float))
        for i in (2, 3):
            v = ref[i, 0]
            if abs(v) < 3e38:
                assert abs(out[i, 0] - v) <= 4e-6 * abs(v)
            else:
                assert np.isinf(out[i, 0]) and np.sign(out[i, 0]) == np.sign(v)
            assert np.all(out[i, 1:] == 0.0)
    ctx.close()
