"""A server's set of SOR fields past the line where its passes go by rows, with sweep counts cut short at different
places, then the rest of it below that line: bit for bit the single solves."""
import numpy as np
import pytest

from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_large_sets_by_rows():
    from paper_2208_02427_gb300 import binding as b
    shapes, caps, dxs = [(4097, 4097), (4096, 4099), (3, 1000), (1025, 700)], [7, 4, 9, 3], [1.0, 0.8, 1.0, 0.8]
    lap = b.Laplace()
    srv = b.Server(lap, hbm_budget=1 << 20, max_running=4, sor_sweeps=4)
    fields, ids, want = [], [], []
    for k, ((m, n), cap, dx) in enumerate(zip(shapes, caps, dxs)):
        psi = wl.random_ring(m, n, 50 + k)
        kw = dict(method="sor", w=1.5 + 0.1 * k, tol=1e-13, max_iter=cap)
        t = b.to_field(psi)
        r = lap.solve(t, dx, 1.0, check_every=4, **kw)
        want.append((t.cpu().numpy(), r["iters"], r["status"]))
        fields.append(b.to_field(psi))
        ids.append(srv.submit(fields[-1], dx=dx, dy=1.0, **kw))
    while sum(srv.step()):
        pass
    res = dict(srv.drain())
    for f, i, (psi, iters, status) in zip(fields, ids, want):
        assert np.array_equal(f.cpu().numpy(), psi)
        assert (res[i]["iters"], res[i]["status"]) == (iters, status)
    srv.close()
    lap.close()
