"""Mixed requests in a server at the sizes where its tails change (all up to 129 points a side, one wider, more of
them than multiprocessors): bit for bit the single solves."""
import numpy as np
import pytest

from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shapes", [[(129, 65), (33, 33)], [(257, 129), (129, 65), (33, 33)],
                                    [(65, 33), (33, 33)] * 80, [(257, 257)] + [(65, 65), (33, 17)] * 80],
                         ids=lambda s: f"{len(s)}x{s[0][0]}")
def test_requests_equal_solves(shapes):
    from paper_2208_02427_gb300 import binding as b
    lap = b.Laplace()
    srv = b.Server(lap, hbm_budget=512 << 20)
    fields, ids = [], []
    for k, (m, n) in enumerate(shapes):
        fields.append(b.to_field(wl.random_ring(m, n, k)))
        ids.append(srv.submit(fields[-1], method="mg_mixed", tol=1e-9))
    while sum(srv.step()):
        pass
    res = dict(srv.drain())
    for k, (m, n) in enumerate(shapes):
        t = b.to_field(wl.random_ring(m, n, k))
        r = lap.solve(t, method="mg_mixed", tol=1e-9)
        assert (res[ids[k]]["iters"], res[ids[k]]["status"]) == (r["iters"], r["status"])
        assert np.array_equal(fields[k].cpu().numpy(), t.cpu().numpy())
    srv.close()
    lap.close()
