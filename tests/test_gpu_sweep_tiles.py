"""Several point sweeps per launch on shared-memory tiles against the one-pass kernels, bit for bit:
sizes on both sides of the rule, uneven tiles, periods that leave every remainder of sweeps per launch,
a pitch wider than the rows, and the stopping rule that needs the last sweep's largest change."""
import numpy as np
import pytest
import torch

from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(65, 65), (97, 70), (70, 301), (513, 385), (1000, 67), (67, 1000), (641, 479), (1531, 1021), (3, 4000)]
METHODS = [("jacobi", 1.0, "paper"), ("sor", 1.7, "paper"), ("gs", 1.0, "paper"), ("sor", 1.7, "diagonal"),
           ("gs", 1.0, "diagonal")]


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


def run(b, lap, psi, method, w, order, dx, every, sweeps, norm="l2_rel"):
    t = b.to_field(psi)
    r = lap.solve(t, dx, 1.0, method=method, w=w, sum_order=order, tol=0.0, check_every=every, max_iter=sweeps,
                  norm=norm)
    torch.cuda.synchronize()
    return t.cpu().numpy(), r


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("method,w,order", METHODS)
def test_tiles_equal_single_passes(b, shape, method, w, order):
    m, n = shape
    psi = wl.random_interior(wl.random_ring(m, n, 3), 4, 1.0)
    lap = b.Laplace()
    for dx in (1.0,) if order == "diagonal" else (1.0, 0.7):
        want, r1 = run(b, lap, psi, method, w, order, dx, 1, 34)
        for every in (2, 5, 17, 32, 34):
            got, r2 = run(b, lap, psi, method, w, order, dx, every, 34)
            assert np.array_equal(got, want), every
            assert r1["r_final"] == r2["r_final"]
    lap.close()


@pytest.mark.parametrize("method,w,order", METHODS)
@pytest.mark.parametrize("norm", ["l2_abs", "maxdelta"])
def test_norms_graphs_and_budgets(b, method, w, order, norm):
    m, n = 257, 193
    psi = wl.random_interior(wl.random_ring(m, n, 5), 6, 1.0)
    field = b.to_field(psi)
    bytes_ = field.stride(0) * n * 8
    outs = []
    for graphs, budget in ((True, 0), (False, 0), (True, bytes_ + (2 << 20)), (True, (2 << 20))):
        if method == "jacobi" and budget == (2 << 20) and bytes_ > budget:
            continue
        lap = b.Laplace(hbm_budget=budget)
        lap.set_graphs(graphs)
        outs.append(run(b, lap, psi, method, w, order, 1.0, 7, 30, norm))
        lap.close()
    lap = b.Laplace()
    want, r = run(b, lap, psi, method, w, order, 1.0, 1, 30, norm)
    lap.close()
    for got, q in outs:
        assert np.array_equal(got, want)
        assert (q["iters"], q["last_check"], q["r_final"]) == (r["iters"], r["last_check"], r["r_final"])


@pytest.mark.parametrize("sweeps", [1, 2, 7, 50])
@pytest.mark.parametrize("room", [0, 300 << 10, 64 << 20])
def test_server_sweeps_equal_single_solves(b, sweeps, room):
    """Fields with a second buffer from the server's pool and fields without (room for none, some, all):
    uneven sizes and spacings, sweep counts cut short at different places, a field solved already."""
    shapes = [(3, 3), (33, 65), (130, 47), (257, 129), (66, 300), (40, 40), (200, 201)]
    lap = b.Laplace()
    srv = b.Server(lap, hbm_budget=room, max_running=len(shapes), sor_sweeps=sweeps)
    fields, ids, want = [], [], []
    for k, (m, n) in enumerate(shapes):
        psi = wl.random_interior(wl.random_ring(m, n, 20 + k), 30 + k, 1.0)
        if k == 5:
            psi[:] = 0.0
        dx, w, cap = (1.0 if k % 2 else 0.8), 1.3 + 0.08 * k, 2 * sweeps + 3 * k
        t = b.to_field(psi)
        r = lap.solve(t, dx, 1.0, method="sor", w=w, tol=1e-13, check_every=sweeps, max_iter=cap)
        want.append((t.cpu().numpy(), r["iters"], r["status"]))
        f = b.to_field(psi)
        fields.append(f)
        ids.append(srv.submit(f, dx=dx, dy=1.0, method="sor", w=w, tol=1e-13, max_iter=cap))
    while sum(srv.step()):
        pass
    res = dict(srv.drain())
    for f, i, (psi, iters, status) in zip(fields, ids, want):
        assert np.array_equal(f.cpu().numpy(), psi)
        assert (res[i]["iters"], res[i]["status"]) == (iters, status)


def test_large_sets_go_pass_by_pass(b):
    """Past the line where the server's sweeps leave the tiles: three fields of over 8 million points in all,
    then two of them alone once the third is done."""
    shapes, caps = [(2049, 2049), (1025, 2049), (2049, 1025)], [4, 9, 9]
    lap = b.Laplace()
    srv = b.Server(lap, hbm_budget=256 << 20, max_running=3, sor_sweeps=4)
    fields, ids, want = [], [], []
    for k, ((m, n), cap) in enumerate(zip(shapes, caps)):
        psi = wl.random_ring(m, n, 50 + k)
        t = b.to_field(psi)
        r = lap.solve(t, method="sor", w=1.9, tol=1e-13, check_every=4, max_iter=cap)
        want.append((t.cpu().numpy(), r["iters"], r["status"]))
        fields.append(b.to_field(psi))
        ids.append(srv.submit(fields[-1], method="sor", w=1.9, tol=1e-13, max_iter=cap))
    while sum(srv.step()):
        pass
    res = dict(srv.drain())
    for f, i, (psi, iters, status) in zip(fields, ids, want):
        assert np.array_equal(f.cpu().numpy(), psi)
        assert (res[i]["iters"], res[i]["status"]) == (iters, status)
