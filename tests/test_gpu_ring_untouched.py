"""The ring of a field is never written, not even with the values it has: while a solve runs, another stream keeps
putting new values into ring points of the field, and finds each as it left it."""
import pytest
import torch

from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

ROUNDS = 250


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


def hammered(field, work):
    """Runs `work` while ring points of the field change on another stream; how many values came back changed."""
    n, m = field.shape
    points = [field[0, m // 3], field[n - 1, m // 2], field[n // 2, 0], field[n // 3, m - 1]]
    log = torch.zeros(ROUNDS, len(points), dtype=torch.float64, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(60_000_000)  # about 30 ms: the work, three times as long, begins while these wait
        for c in range(ROUNDS):
            for p in points:
                p.fill_(1.0 + c)
            torch.cuda._sleep(20_000)
            for k, p in enumerate(points):
                log[c, k].copy_(p)
    work()
    torch.cuda.synchronize()
    want = 1.0 + torch.arange(ROUNDS, dtype=torch.float64, device="cuda")[:, None]
    left = torch.stack(points)
    return int((log != want).sum()) + int((left != float(ROUNDS)).sum())


@pytest.mark.parametrize("method,order", [("sor", "paper"), ("sor", "diagonal"), ("gs", "paper"), ("jacobi", "paper")])
@pytest.mark.parametrize("sweeps", [60000, 60001])
def test_solve(b, method, order, sweeps):
    lap = b.Laplace()
    t = b.to_field(wl.random_ring(257, 193, 3))
    kw = dict(method=method, w=1.5, sum_order=order, tol=0.0, check_every=30)
    lap.solve(t, max_iter=60, **kw)  # the plan and graph
    assert hammered(t, lambda: lap.solve(t, max_iter=sweeps, **kw)) == 0
    lap.close()


def test_server(b):
    lap = b.Laplace()
    srv = b.Server(lap, hbm_budget=16 << 20, max_running=4, sor_sweeps=20000)
    t = b.to_field(wl.random_ring(257, 193, 3))
    srv.submit(t, method="sor", w=1.5, tol=0.0, max_iter=80000)
    srv.step()

    def steps():
        while sum(srv.step()):
            pass

    assert hammered(t, steps) == 0
    srv.close()
    lap.close()
