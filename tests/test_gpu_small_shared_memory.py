"""One-CTA solves whose arrays end just below 48 KB, where the kernels' static arrays take them past what a
launch may have unasked: every size up to that line and a few past it runs, as the oracle does."""
import numpy as np
import pytest
import torch

import oracle as ora
from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


# 16 bytes a point in Jacobi's two fields: 2981 .. 3090 points about the line of 3072
@pytest.mark.parametrize("shape", [(11, 271), (54, 55), (55, 55), (3, 1000), (48, 63), (51, 60), (3, 1024), (64, 48),
                                   (439, 7), (30, 103)])
def test_jacobi(b, shape):
    psi = wl.random_interior(wl.random_ring(*shape, 5), 9, 1.0)
    lap = b.Laplace()
    t = b.to_field(psi)
    g = lap.solve(t, method="jacobi", norm="maxdelta", tol=0.0, max_iter=3)
    u, o = ora.solve(psi, ora.JACOBI, dx=1.0, dy=1.0, tol=0.0, norm=ora.NORM_MAXDELTA, max_iter=3, check_every=1)
    assert (g["iters"], g["status"]) == (o["iters"], o["status"])
    assert np.array_equal(t.cpu().numpy(), u)
    lap.close()


# the lines' work space and tables come on top of two fields: 2180 .. 2480 points about the line, wherever it
# lies for the method
@pytest.mark.parametrize("method,form", [("adi", "A"), ("adi", "B"), ("slor", "A"), ("slor", "B")])
@pytest.mark.parametrize("n", [38, 42, 45, 48, 50])
def test_lines(b, method, form, n):
    lap = b.Laplace()
    for m in range(2180 // n, 2480 // n + 1):
        psi = wl.random_interior(wl.random_ring(m, n, 5), 9, 1.0)
        t = b.to_field(psi)
        g = lap.solve(t, method=method, w=1.25, line_form=form, norm="maxdelta", tol=0.0, max_iter=1)
        want, o = ora.solve(psi, ora.ADI if method == "adi" else ora.SLOR, dx=1.0, dy=1.0, w=1.25,
                            form=ora.FORM_A if form == "A" else ora.FORM_B, tol=0.0, norm=ora.NORM_MAXDELTA,
                            max_iter=1, check_every=1)
        assert g["iters"] == o["iters"] == 1, (m, n)
        # the bar of the one-CTA line solves
        assert np.max(np.abs(t.cpu().numpy() - want)) <= 1e-12 * max(1.0, np.max(np.abs(want))), (m, n)
    torch.cuda.synchronize()
    lap.close()


# the lexicographic solves' one field: 6127 .. 6160 points about the line of 6144
@pytest.mark.parametrize("shape", [(11, 557), (64, 96), (3, 2045), (3, 2048), (61, 101), (88, 70)])
@pytest.mark.parametrize("method,w", [("gs_lex", 1.0), ("sor_lex", 1.4)])
def test_lexicographic(b, shape, method, w):
    psi = wl.random_interior(wl.random_ring(*shape, 5), 9, 1.0)
    lap = b.Laplace()
    t = b.to_field(psi)
    g = lap.solve(t, method=method, w=w, norm="maxdelta", tol=0.0, max_iter=2)
    u, o = ora.solve(psi, ora.GS if w == 1.0 else ora.SOR, ordering=ora.LEX, w=w, dx=1.0, dy=1.0, tol=0.0,
                     norm=ora.NORM_MAXDELTA, max_iter=2, check_every=1)
    assert g["iters"] == o["iters"]
    assert np.array_equal(t.cpu().numpy(), u)
    lap.close()
