"""Line solves against the oracle where their layout changes: lines on both sides of the 48 KB of shared
memory that need no attribute, few and many lines to a CTA, chunks shorter than the boundary layer, rows by
the row kernel and by a thread per chunk (1024 unknowns, and without room for its scratch)."""
import numpy as np
import pytest

import oracle as ora
from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(5950, 5), (6000, 5), (6090, 5), (5, 6000), (1026, 40), (1027, 40), (16000, 7), (7, 9000), (157, 11),
          (11, 157), (320, 1290), (1290, 320), (615, 611), (129, 70), (64, 1021)]


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


def solve(b, psi, method, form, w, dx, budget=0):
    lap = b.Laplace(hbm_budget=budget)
    t = b.to_field(psi)
    r = lap.solve(t, dx, 1.0, method=method, w=w, line_form=form, tol=0.0, max_iter=2, check_every=2)
    lap.close()
    return t.cpu().numpy(), r


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("method,form,w,dx", [("slor", "A", 1.3, 1.0), ("slor", "B", 1.25, 0.8), ("adi", "A", 1.0, 1.0),
                                              ("adi", "B", 1.3, 1.25)])
def test_line_solves(b, shape, method, form, w, dx):
    m, n = shape
    psi = wl.random_interior(wl.random_ring(m, n, 5 + m), 9 + n, 1.0)
    got, r = solve(b, psi, method, form, w, dx)
    want, o = ora.solve(psi, ora.ADI if method == "adi" else ora.SLOR, dx=dx, dy=1.0, w=w,
                        form=ora.FORM_A if form == "A" else ora.FORM_B, tol=0.0, max_iter=2, check_every=2)
    # four half sweeps at most of exact line solves whose matrices' condition is at most 15 (dx = 1.25 along
    # y): a few ulp each
    assert np.max(np.abs(got - want)) <= 1e-13 * max(1.0, np.max(np.abs(want)))
    assert abs(r["r_final"] - o["r_final"]) <= 1e-12 * o["r0"]


@pytest.mark.parametrize("method", ["slor", "adi"])
def test_rows_without_scratch(b, method):
    m, n = 801, 1201
    psi = wl.random_interior(wl.random_ring(m, n, 3), 4, 1.0)
    # room for the arena, the flags and the tables (and the columns' scratch), not for the rows'
    tight = (1 << 20) * (3 if method == "slor" else 3 + 8)
    got, _ = solve(b, psi, method, "A", 1.2, 1.0, budget=tight)
    want, _ = solve(b, psi, method, "A", 1.2, 1.0)
    assert np.max(np.abs(got - want)) <= 1e-13
