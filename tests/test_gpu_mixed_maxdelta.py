"""The mixed solver under the paper's stopping rule (Eq. 16): one test per check period, the same solve with the
loop on the device as with launches from the host."""
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


@pytest.mark.parametrize("shape,dx", [((65, 33), 1.0), ((193, 129), 1.0), ((97, 65), 0.7)])
@pytest.mark.parametrize("tol,every,cap", [(0.0, 1, 10), (0.0, 1, 7), (0.0, 2, 6), (0.0, 3, 7), (1e-9, 1, 50),
                                           (1e-9, 2, 51), (1e-3, 1, 50), (np.inf, 2, 8)])
def test_graphs_equal_launches(b, shape, dx, tol, every, cap):
    psi = wl.random_ring(*shape, seed=11)
    out = []
    for graphs in (False, True):
        lap = b.Laplace()
        lap.set_graphs(graphs)
        t = b.to_field(psi)
        r = lap.solve(t, dx, 1.0, method="mg_mixed", norm="maxdelta", tol=tol, check_every=every, max_iter=cap)
        torch.cuda.synchronize()
        out.append((t.cpu().numpy(), r))
        lap.close()
    (want, r0), (got, r1) = out
    assert (r1["iters"], r1["status"], r1["last_check"]) == (r0["iters"], r0["status"], r0["last_check"])
    assert np.array_equal(got, want)
    assert r1["r_final"] == r0["r_final"]
    if tol == 0.0:
        assert r1["iters"] == cap


def test_change_of_the_last_cycle(b):
    """last_check is the largest change that the last cycle made."""
    m, n = 129, 65
    psi = wl.random_ring(m, n, seed=4)
    fields = []
    lap = b.Laplace()
    for cap in (2, 3):
        t = b.to_field(psi)
        r = lap.solve(t, method="mg_mixed", norm="maxdelta", tol=0.0, max_iter=cap)
        assert (r["iters"], r["status"]) == (cap, "max_iter")
        fields.append(t.cpu().numpy())
    assert r["last_check"] == np.max(np.abs(fields[1] - fields[0]))
    lap.close()
