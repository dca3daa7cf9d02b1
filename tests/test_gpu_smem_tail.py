"""The small-level tail in shared memory (one CTA, or a cluster splitting its first levels by rows)
against the cycle run level by level: the same iterates bit for bit, at sizes where the split changes
(number of split levels, CTAs without rows, uneven last blocks), for odd coarsest levels (more than
32 unknowns), dx != dy, 1/d = 1/2, SOR smoothers and missing sweeps, and fields with zero or subnormal
regions, whose black residuals are not the exact zeros that Gauss-Seidel leaves elsewhere."""
import numpy as np
import pytest
import torch

from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(33, 33), (31, 33), (33, 31), (65, 17), (17, 65), (97, 65), (49, 193), (257, 129), (113, 225), (129, 257),
          (41, 21), (61, 57), (513, 65), (81, 401)]


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


def solve(b, lap, x, dx, **kw):
    f = b.to_field(x)
    r = lap.solve(f, dx, 1.0, tol=0.0, max_iter=2, **kw)
    torch.cuda.synchronize()
    return f.cpu().numpy().copy(), r["r_final"]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("method", ["mg", "mg_mixed", "mg_fp32"])
@pytest.mark.parametrize("kw", [dict(), dict(dx=0.7), dict(dx=1e-9), dict(smoother_w=1.2, nu1=1, nu2=3),
                                dict(nu1=0, nu2=2), dict(nu1=2, nu2=0)])
def test_tail_equals_levels(b, shape, method, kw):
    kw = dict(kw)
    dx = kw.pop("dx", 1.0)
    lap = b.Laplace()
    x = wl.random_ring(*shape, seed=7 * shape[0] + shape[1])
    want = solve(b, lap, x, dx, method=method, tail_size=-1, **kw)
    for tail in (0, 17, 65, max(shape)):
        got = solve(b, lap, x, dx, method=method, tail_size=tail, **kw)
        assert np.array_equal(got[0], want[0], equal_nan=True), tail
        assert got[1] == want[1] or (np.isnan(got[1]) and np.isnan(want[1]))
    lap.close()


@pytest.mark.parametrize("scale", [1e-305, 1e-310, 0.0])
def test_underflow(b, scale):
    """Values so small that a quarter of a neighbour sum is subnormal."""
    lap = b.Laplace()
    x = wl.random_ring(65, 65, seed=2) * scale
    x[0, 3] = 1e-300
    want = solve(b, lap, x, 1.0, method="mg", tail_size=-1)
    got = solve(b, lap, x, 1.0, method="mg", tail_size=65)
    assert np.array_equal(got[0], want[0])
    lap.close()
