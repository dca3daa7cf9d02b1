"""The mixed solver's residual where a run's values (62 columns by 8 rows) span many binades: a ring point far above
the others, and fields that fall off beside an edge. The residual is the exact one rounded to FP32 whatever its run
holds, so its norm close to the solution is that of the returned field to FP32 accuracy."""
import math

import numpy as np
import pytest
import torch

from paper_2208_02427_gb300 import workloads as wl
from tests.test_gpu_residual32_small import exact_norm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


def ring(m, n, kind):
    if kind[0] == "hot":  # one value of 2^p on the bottom or left edge, the others 1/4 .. 1
        psi = wl.random_ring(m, n, 3)
        psi[psi != 0.0] = 0.25 + 0.75 * psi[psi != 0.0]
        psi[(0, m // 3) if kind[2] == 0 else (n // 2, 0)] = 2.0 ** kind[1]
        return psi
    psi = np.zeros((n, m))  # half a sine on the left or bottom edge: falls off by e^-pi in n or m points
    if kind[1] == 0:
        psi[1:-1, 0] = np.sin(math.pi * np.arange(1, n - 1) / (n - 1))
    else:
        psi[0, 1:-1] = np.sin(math.pi * np.arange(1, m - 1) / (m - 1))
    return psi


KINDS = [("hot", p, edge) for p in (4, 10, 20, 27) for edge in (0, 1)] + [("mode", 0), ("mode", 1)]


@pytest.mark.parametrize("shape", [(129, 65), (65, 129), (193, 33), (33, 193), (65, 17)])
@pytest.mark.parametrize("kind", KINDS, ids=lambda k: "-".join(map(str, k)))
def test_norm_near_the_solution(b, shape, kind):
    m, n = shape
    psi = ring(m, n, kind)
    lap = b.Laplace()
    t = b.to_field(psi)
    r = lap.solve(t, method="mg_mixed", tol=0.0, norm="l2_abs", max_iter=14)
    torch.cuda.synchronize()
    got = t.cpu().numpy()
    want = exact_norm(got)
    # each residual rounds at 2^-24, its square too, and a lane sums up to some sixty of them in FP32
    assert abs(r["last_check"] - want) <= 1e-5 * want
    f = b.to_field(psi)
    s = lap.solve_batched([f], method="mg_mixed", tol=0.0, norm="l2_abs", max_iter=14)
    assert np.array_equal(f.cpu().numpy(), got)
    assert abs(s[0]["r_final"] - want) <= 1e-5 * want
    lap.close()


@pytest.mark.parametrize("exponent", [-56, -40, 0, 100, 111])
def test_range_at_the_ends_of_the_scale(b, exponent):
    """A wide run at magnitudes where its FP32 results come near the ends of their range, and past the line from
    which such runs take the FP64 expression: the solve scales with the field."""
    m, n = 129, 33
    psi = ring(m, n, ("hot", 5, 0))
    lap = b.Laplace()
    t, u = b.to_field(psi), b.to_field(np.ldexp(psi, exponent))
    r = lap.solve(t, method="mg_mixed", tol=0.0, norm="l2_abs", max_iter=9)
    q = lap.solve(u, method="mg_mixed", tol=0.0, norm="l2_abs", max_iter=9)
    want = exact_norm(np.ldexp(u.cpu().numpy(), -exponent))
    got = q["last_check"] * 2.0 ** -exponent
    # the fixed-point sums run while r0 is within 2^-100 .. 2^100 and no value is too small for them; else, after
    # nine cycles, the residual is some 1e-12 of r0 and FP64's rounding of it 1e-3 of that at most
    exact = -40 <= exponent and q["r0"] < 2.0 ** 100
    assert abs(got - want) <= (1e-5 if exact else 1e-2) * want
    assert abs(r["last_check"] - want) <= 1e-1 * want
    lap.close()
