"""Columns of fields past the L2's size, where form A cuts them into more chunks: a half sweep of both forms against
an exact elimination of every line in numpy."""
import numpy as np
import pytest

from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def zebra_columns(psi, w, b2, form):
    """Odd columns, then even ones, by the Thomas algorithm over all lines of a colour at once."""
    u = psi.copy()
    n = u.shape[0] - 2
    d = 2.0 * (1.0 + b2)
    off = b2 if form == "A" else w * b2
    for first in (1, 2):
        x = u[:, first:-1:2]
        rhs = u[1:-1, first - 1:-2:2] + u[1:-1, first + 1::2]
        if form == "B":
            rhs = w * rhs + d * (1.0 - w) * x[1:-1]
        rhs[0] += off * x[0]
        rhs[-1] += off * x[-1]
        c = np.empty(n)
        den = d
        for k in range(n):
            if k:
                den = d - off * c[k - 1]
                rhs[k] += off * rhs[k - 1]
            c[k] = off / den
            rhs[k] /= den
        for k in range(n - 2, -1, -1):
            rhs[k] += c[k] * rhs[k + 1]
        x[1:-1] = rhs if form == "B" else w * rhs + (1.0 - w) * x[1:-1]
    return u


@pytest.mark.parametrize("m,n", [(4097, 4097), (3300, 3300), (1100, 10001)])
@pytest.mark.parametrize("form", ["A", "B"])
def test_half_sweep(m, n, form):
    from paper_2208_02427_gb300 import binding as b
    psi = wl.random_interior(wl.random_ring(m, n, 3), 4, 1.0)
    lap = b.Laplace()
    t = b.to_field(psi)
    lap.line_sweep(t, 1.2, form, 1, dx=0.9, dy=1.0)
    want = zebra_columns(psi, 1.2, 0.81, form)
    # the repository's bar for line solves: a few ulp times the line matrix' condition (13 at most here), twice
    assert np.max(np.abs(t.cpu().numpy() - want)) <= 1e-12
    lap.close()
