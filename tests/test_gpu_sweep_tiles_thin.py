"""Thin grids, whose diagonal sweeps go one to a launch on tiles: an odd number of them ends with a launch that
only copies. Bit for bit the one-pass kernels."""
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


@pytest.mark.parametrize("shape", [(3, 59200), (59200, 3), (5, 50000), (50000, 5)])
@pytest.mark.parametrize("norm,every,sweeps", [("l2_rel", 3, 6), ("maxdelta", 4, 10), ("l2_rel", 4, 7)])
def test_one_sweep_a_launch(b, shape, norm, every, sweeps):
    psi = wl.random_interior(wl.random_ring(*shape, 3), 4, 1.0)
    lap = b.Laplace()
    out = []
    for period in (1, every):
        t = b.to_field(psi)
        r = lap.solve(t, method="sor", w=1.7, sum_order="diagonal", tol=0.0, check_every=period, max_iter=sweeps,
                      norm=norm)
        torch.cuda.synchronize()
        out.append((t.cpu().numpy(), (r["iters"], r["last_check"], r["r_final"])))
    assert np.array_equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]
    lap.close()
