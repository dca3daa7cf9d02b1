"""The configuration that a batch's size gives (tail, tiles, more small tails than multiprocessors): the values of
the cycle run without a tail and one kernel per pass, bit for bit, on both sides of its lines."""
import pytest
import torch

from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


SETS = [[(33, 33)], [(65, 33), (65, 65)], [(129, 129), (65, 33), (9, 9)], [(65, 65), (33, 17)] * 80,
        [(33, 33)] * 320, [(129, 65)] * 12, [(129, 33), (65, 65)] * 90, [(257, 129), (33, 33), (65, 65)], [(33, 33)] * 2500]


@pytest.mark.parametrize("shapes", SETS, ids=lambda s: f"{len(s)}x{s[0][0]}")
@pytest.mark.parametrize("kw", [dict(method="mg"), dict(method="mg_mixed"), dict(method="mg_mixed", nu1=4, nu2=4),
                                dict(method="mg_mixed", unfused=True), dict(method="mg_mixed", tiling=1)],
                         ids=lambda kw: "-".join(map(str, kw.values())))
def test_values(b, shapes, kw):
    lap = b.Laplace()
    pitch = max(m for m, _ in shapes)
    rows = sum(n for _, n in shapes)
    start = torch.rand(rows, pitch, dtype=torch.float64, generator=torch.Generator().manual_seed(4)).cuda()
    out = []
    for forced in (dict(), dict(tail_size=-1, **({} if kw["method"] == "mg" else {"unfused": True}))):
        buf, at, fields = start.clone(), 0, []
        for m, n in shapes:
            fields.append(buf[at:at + n, :m])
            at += n
        res = lap.solve_batched(fields, method=kw["method"], tol=1e-8, max_iter=3,
                                **{**{k: v for k, v in kw.items() if k != "method"}, **forced})
        torch.cuda.synchronize()
        out.append((buf, [(r["iters"], r["r_final"]) for r in res]))
    assert torch.equal(out[0][0], out[1][0])
    assert out[0][1] == out[1][1]
    lap.close()


def test_small_grids_get_a_tail(b):
    lap = b.Laplace()
    for count, kw, tail in ((2, dict(method="mg"), 65), (2, dict(method="mg_mixed"), 65),
                            (200, dict(method="mg_mixed", unfused=True), 65), (2000, dict(method="mg_mixed"), -1)):
        lap.solve_batched([b.to_field(wl.random_ring(33, 33, 1)) for _ in range(count)], tol=1e-6, **kw)
        assert lap.last_batch_config()["tail_size"] == tail, (count, kw)
    lap.close()
