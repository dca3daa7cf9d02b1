"""Device memory that a handle holds beside its scratch: bounded, and by the grid's own size, not by its pitch."""
import pytest
import torch

from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SLACK = 24 << 20  # the allocator's rounding, graphs, kernels loaded on first use


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


def held(b, lap, t, **kw):
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    lap.solve(t, **kw)
    torch.cuda.synchronize()
    return before - torch.cuda.mem_get_info()[0]


def test_wide_pitch(b):
    """The second field of the tile sweeps takes a pitch of its own: 257 x 193 points in rows of 200,000."""
    m, n, pitch = 257, 193, 200_000
    buf = torch.zeros(n, pitch, dtype=torch.float64, device="cuda")
    psi = wl.random_ring(m, n, 3)
    lap = b.Laplace()
    t = buf[:, :m]
    kw = dict(method="sor", w=1.7, tol=0.0, check_every=20, max_iter=41)
    lap.solve(b.to_field(wl.random_ring(33, 33, 1)), **kw)  # kernels loaded, the handle's first blocks
    t.copy_(torch.as_tensor(psi))
    assert held(b, lap, t, **kw) <= m * n * 8 * 2 + SLACK
    want = b.to_field(psi)
    lap.solve(want, **dict(kw, check_every=1))
    assert torch.equal(t, want)
    lap.close()


@pytest.mark.parametrize("m,n", [(1026, 16385), (1026, 4001), (400, 16000)])
def test_rows(b, m, n):
    """Rows by threads hold at most 64 MiB of scratch beside the columns' own."""
    f = b.field(m, n)
    f.zero_()
    f[0] = 1.0
    lap = b.Laplace()
    lap.solve(b.to_field(wl.random_ring(33, 33, 1)), method="adi", w=1.2, max_iter=2)
    kw = dict(method="adi", w=1.2, tol=0.0, max_iter=2, check_every=2)
    columns = ((m - 1) // 2 + 32) * (n - 2) * 8
    assert held(b, lap, f, **kw) <= lap.workspace_bytes(f, **kw) + columns + (64 << 20) + SLACK
    lap.close()
