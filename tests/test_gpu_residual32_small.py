"""The mixed solver's residual close to the solution, where it is a few units in the last place of the field: its
norm is that of the returned field, taken in whole numbers, to FP32 accuracy. (Fields within three binades of
their largest value, for which the fixed-point sums cut nothing.)"""
import math

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


def exact_norm(psi):
    """||(E + W) + (N + S) - 4 C||_2 in whole numbers."""
    mant, e = np.frexp(psi)
    lo = int(e[mant != 0.0].min()) - 53
    shift = np.where(mant != 0.0, e - 53 - lo, 0)
    v = np.array([int(a) << int(s) for a, s in zip(np.ldexp(mant, 53).ravel(), shift.ravel())],
                 dtype=object).reshape(psi.shape)
    r = v[1:-1, 2:] + v[1:-1, :-2] + v[2:, 1:-1] + v[:-2, 1:-1] - 4 * v[1:-1, 1:-1]
    total = int((r * r).sum())
    cut = max(0, total.bit_length() - 120) // 2
    return math.ldexp(math.sqrt(float(total >> 2 * cut)), lo + cut)


@pytest.mark.parametrize("shape", [(129, 65), (65, 129), (193, 33), (33, 193), (65, 17), (17, 9)])
@pytest.mark.parametrize("cycles", [3, 10, 12, 14])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_norm_near_the_solution(b, shape, cycles, sign):
    m, n = shape
    psi = wl.random_ring(m, n, 3)
    edge = np.ones((n, m), dtype=bool)
    edge[1:-1, 1:-1] = False
    psi[edge] = sign * (0.25 + 0.75 * psi[edge])
    lap = b.Laplace()
    t = b.to_field(psi)
    r = lap.solve(t, method="mg_mixed", tol=0.0, norm="l2_abs", max_iter=cycles)
    torch.cuda.synchronize()
    got = t.cpu().numpy()
    want = exact_norm(got)
    # each residual rounds at 2^-24, its square too, and a lane sums up to some sixty of them in FP32
    assert abs(r["last_check"] - want) <= 1e-5 * want
    f = b.to_field(psi)
    s = lap.solve_batched([f], method="mg_mixed", tol=0.0, norm="l2_abs", max_iter=cycles)
    assert np.array_equal(f.cpu().numpy(), got)
    assert abs(s[0]["r_final"] - want) <= 1e-5 * want
    lap.close()
