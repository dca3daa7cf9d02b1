"""Whole solves in one CTA at the sizes where their layout changes: one line, one unknown, as many
lanes as unknowns, a short last chunk, the 4096-point limit. Point methods are the oracle's bit for
bit; line methods to rounding (they reassociate)."""
import numpy as np
import pytest
import torch

import oracle as ora
from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

# lines of 1 .. 1363 unknowns and 1 .. 1363 lines: 2 to 32 lanes a line, no chunk, chunks of one
# and of hundreds of unknowns, last chunks shorter than the others
SHAPES = [(3, 3), (3, 4), (4, 3), (3, 1365), (1365, 3), (64, 64), (63, 65), (34, 33), (35, 35), (10, 200),
          (500, 7), (18, 18), (19, 17), (129, 31)]


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


def field(m, n):
    return wl.random_interior(wl.random_ring(m, n, 5 + m), 9 + n, 1.0)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("method,form", [("adi", "A"), ("adi", "B"), ("slor", "A"), ("slor", "B")])
@pytest.mark.parametrize("beta", [1.0, 0.6])
def test_line_solves(b, shape, method, form, beta):
    m, n = shape
    lap = b.Laplace()
    psi = field(m, n)
    t = b.to_field(psi)
    g = lap.solve(t, beta, 1.0, method=method, w=1.25, line_form=form, norm="maxdelta", tol=0.0,
                  check_every=2, max_iter=5)
    want, o = ora.solve(psi, ora.ADI if method == "adi" else ora.SLOR, dx=beta, dy=1.0, w=1.25,
                        form=ora.FORM_A if form == "A" else ora.FORM_B, tol=0.0,
                        norm=ora.NORM_MAXDELTA, max_iter=5, check_every=2)
    got = t.cpu().numpy()
    assert (g["iters"], g["status"]) == (o["iters"], o["status"])
    # the repository's bar for line solves: 10 half sweeps of exact solves, each a few ulp times the
    # line matrix' condition (23 at most here, beta = 0.6 form B), about 3e-13
    assert np.max(np.abs(got - want)) <= 1e-12 * max(1.0, np.max(np.abs(want)))
    assert abs(g["r0"] - o["r0"]) <= 1e-13 * o["r0"]
    assert abs(g["r_final"] - o["r_final"]) <= 1e-11 * o["r0"]
    lap.close()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("method,w", [("jacobi", 1.0), ("gs", 1.0), ("sor", 1.6)])
@pytest.mark.parametrize("beta", [1.0, 0.6])
def test_point_solves(b, shape, method, w, beta):
    m, n = shape
    lap = b.Laplace()
    psi = field(m, n)
    t = b.to_field(psi)
    g = lap.solve(t, beta, 1.0, method=method, w=w, norm="maxdelta", tol=0.0, check_every=2, max_iter=5)
    kw = {"jacobi": dict(method=ora.JACOBI), "gs": dict(method=ora.GS, ordering=ora.RB),
          "sor": dict(method=ora.SOR, ordering=ora.RB, w=w)}[method]
    u, o = ora.solve(psi, dx=beta, dy=1.0, tol=0.0, norm=ora.NORM_MAXDELTA, max_iter=5, check_every=2, **kw)
    assert (g["iters"], g["status"]) == (o["iters"], o["status"])  # one unknown stops changing at once
    assert np.array_equal(t.cpu().numpy(), u)
    # the residual norms are the multi-CTA norm kernels' bit for bit
    assert g["r0"] == lap.residual(b.to_field(psi), beta, 1.0)
    assert g["r_final"] == lap.residual(t, beta, 1.0)
    torch.cuda.synchronize()
    lap.close()


def test_not_finite_and_loose_tolerances(b):
    """A NaN in the interior stops at once, an overflowing iterate at its test, a tolerance of
    infinity after the first test."""
    lap = b.Laplace()
    for method in ("sor", "jacobi", "adi", "slor"):
        psi = field(25, 17)
        psi[5, 5] = np.nan
        g = lap.solve(b.to_field(psi), method=method, w=1.2, norm="maxdelta", tol=1e-9, max_iter=50)
        assert g["status"] == "diverged" and g["iters"] == 0
        g = lap.solve(b.to_field(field(25, 17)), method=method, w=1.2, norm="maxdelta", tol=np.inf,
                      check_every=3, max_iter=50)
        assert g["status"] == "converged" and g["iters"] == 3
    lap.close()
