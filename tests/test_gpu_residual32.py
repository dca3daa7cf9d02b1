"""The mixed solver's residual on the integer pipe: its norm against the FP64 residual at the edges of its
runs (62 columns by 8 rows), at magnitudes on both sides of its range, on rows that are not 16-byte
aligned, and with values that take the FP64 expression."""
import numpy as np
import pytest
import torch

from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(3, 3), (9, 10), (33, 11), (64, 17), (65, 9), (66, 18), (129, 129), (257, 65), (65, 257), (513, 513)]


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


def norm(psi):
    r = psi[1:-1, 2:] + psi[1:-1, :-2] + psi[2:, 1:-1] + psi[:-2, 1:-1] - 4.0 * psi[1:-1, 1:-1]
    return float(np.sqrt(np.sum(r * r)))


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("exponent", [0, -52, -80, 100])
@pytest.mark.parametrize("odd", [False, True])
def test_norm_after_a_cycle(b, shape, exponent, odd):
    m, n = shape
    psi = np.ldexp(wl.random_interior(wl.random_ring(m, n, 7), 8, 1.0), exponent)
    lap = b.Laplace()
    buf = torch.zeros(n, m + 5 + (m % 2 == 1), dtype=torch.float64, device="cuda")  # an odd or an even pitch
    t = buf[:, 1:m + 1] if odd else b.to_field(psi)
    t.copy_(torch.as_tensor(psi))
    r = lap.solve(t, method="mg_mixed", tol=0.0, norm="l2_abs", max_iter=1)
    got = t.cpu().numpy()
    want = norm(got)
    # per point 2^-52 of the run's largest value before the rounding to FP32 (about 4 for these fields, in
    # units of 2^exponent), FP32 rounding of residuals and squares (2^-24 each, 4 sums deep at the least);
    # numpy's own residual rounds at 2^-50
    floor = np.sqrt(m * n) * 4.0 * 2.0 ** (exponent - 49)
    assert abs(r["last_check"] - want) <= 1e-5 * want + floor
    lap.close()


@pytest.mark.parametrize("exponent", [-90, -64, -60, -30, 40, 95])
def test_scaling_by_powers_of_two(b, exponent):
    psi = wl.random_ring(257, 129, 3)
    lap = b.Laplace()
    t, u = b.to_field(psi), b.to_field(np.ldexp(psi, exponent))
    r, q = lap.solve(t, method="mg_mixed", tol=1e-10), lap.solve(u, method="mg_mixed", tol=1e-10)
    assert (r["status"], r["iters"]) == (q["status"], q["iters"]) == ("converged", r["iters"])
    a, c = t.cpu().numpy(), np.ldexp(u.cpu().numpy(), -exponent)
    # both stop at a residual of 1e-10 r0: errors of at most about n^2/4 times that a point
    assert np.max(np.abs(a - c)) <= 1e-9
    lap.close()


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e300])
def test_values_outside_the_range(b, value):
    psi = wl.random_ring(129, 65, 3)
    psi[0, 0] = value  # a corner belongs to no stencil
    lap = b.Laplace()
    t = b.to_field(psi)
    r = lap.solve(t, method="mg_mixed", tol=1e-10)
    assert r["status"] == "converged"
    psi[0, 40] = value
    u = b.to_field(psi)
    fields = [b.to_field(psi), b.to_field(wl.random_ring(65, 65, 4))]
    q = lap.solve(u, method="mg_mixed", tol=1e-10, max_iter=20)
    s = lap.solve_batched(fields, 1.0, 1.0, method="mg_mixed", tol=1e-10, max_iter=20)
    assert s[0]["status"] == q["status"] and s[1]["status"] == "converged"
    assert np.array_equal(u.cpu().numpy(), fields[0].cpu().numpy(), equal_nan=True)
    lap.close()
