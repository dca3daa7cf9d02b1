"""The row streams below FP32's normal range, where a product by 0.5 or 0.25 rounds: the same values as the
per-pass kernels, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


@pytest.mark.parametrize("scale", [1e-30, 1e-37, 1e-38, 1e-40, 1e-42, 1e-44])
@pytest.mark.parametrize("shape", [(33, 33), (65, 17), (129, 65), (9, 321), (257, 513)])
@pytest.mark.parametrize("kw", [{}, {"nu1": 3, "nu2": 3}, {"smoother_w": 1.1}, {"dx": 0.7},
                                {"dx": 0.7, "smoother_w": 0.9, "inner_cycles": 2}], ids=str)
def test_streams_equal_passes(b, shape, scale, kw):
    kw = dict(kw)
    dx = kw.pop("dx", 1.0)
    psi = wl.random_ring(*shape, seed=3) * scale
    lap = b.Laplace()
    want = b.to_field(psi)
    lap.solve(want, dx, 1.0, method="mg_mixed", tol=0.0, max_iter=2, tail_size=-1, unfused=True, **kw)
    single = b.to_field(psi)
    lap.solve(single, dx, 1.0, method="mg_mixed", tol=0.0, max_iter=2, tail_size=-1, **kw)
    batch = [b.to_field(psi) for _ in range(3)]
    lap.solve_batched(batch, dx, 1.0, method="mg_mixed", tol=0.0, max_iter=2, tail_size=-1, **kw)
    torch.cuda.synchronize()
    want = want.cpu().numpy()
    assert np.any(want[1:-1, 1:-1] != 0.0) or scale < 1e-43
    for t in [single, *batch]:
        assert np.array_equal(t.cpu().numpy(), want)
    lap.close()
