"""The FP32 levels' row streams against the cycle run one kernel per pass: the same expressions, so
the same bits, at the sizes where the streams' cut changes -- widths around one and two column
blocks (128 columns, 116 or 120 owned), segments of 4, 8 and 16 lanes, strips that end inside a
segment -- for every smoothing count they cover, and for fields whose rows are not 16-byte aligned."""
import numpy as np
import pytest
import torch

from paper_2208_02427_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(113, 49), (117, 49), (121, 97), (125, 33), (129, 41), (133, 65), (241, 33), (245, 49), (249, 57),
          (253, 65), (257, 73), (361, 81), (65, 129), (61, 201), (33, 401), (29, 257), (13, 129), (9, 9), (1025, 513)]


@pytest.fixture(scope="module")
def b():
    from paper_2208_02427_gb300 import binding
    binding.load()
    return binding


def solve(b, lap, f, dx, **kw):
    r = lap.solve(f, dx, 1.0, method="mg_mixed", tol=0.0, max_iter=2, **kw)
    torch.cuda.synchronize()
    return f.cpu().numpy().copy(), r


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("nu,w,dx", [((2, 2), 1.0, 1.0), ((2, 2), 1.2, 0.7), ((1, 3), 1.0, 0.7), ((3, 1), 1.2, 1.0)])
@pytest.mark.parametrize("inner", [1, 2])
def test_streams_equal_passes(b, shape, nu, w, dx, inner):
    lap = b.Laplace()
    x = wl.random_ring(*shape, seed=31 * shape[0] + shape[1])
    kw = dict(nu1=nu[0], nu2=nu[1], smoother_w=w, inner_cycles=inner, tail_size=-1)
    want, r0 = solve(b, lap, b.to_field(x), dx, unfused=True, **kw)
    got, r1 = solve(b, lap, b.to_field(x), dx, **kw)
    assert np.array_equal(got, want)
    assert r0["r_final"] == r1["r_final"]
    lap.close()


@pytest.mark.parametrize("shift,pad", [(1, 7), (0, 1), (1, 0)])
def test_unaligned_fields(b, shift, pad):
    """Rows at 8 mod 16 bytes and odd pitches take the update's scalar path."""
    lap = b.Laplace()
    m, n = 257, 129
    x = wl.random_ring(m, n, seed=8)
    want, _ = solve(b, lap, b.to_field(x), 1.0, unfused=True)
    f = torch.zeros(n, m + shift + pad, dtype=torch.float64, device="cuda")[:, shift:shift + m]
    f.copy_(torch.as_tensor(x))
    got, _ = solve(b, lap, f, 1.0)
    assert np.array_equal(got, want)
    lap.close()


@pytest.mark.parametrize("inner", [1, 2])
def test_batched_streams(b, inner):
    """Every shape in one batch, pieces of many problems in one launch, with and without a tail."""
    lap = b.Laplace()
    inputs = [wl.random_ring(m, n, seed=5 + m + n) for m, n in SHAPES]
    dx = [1.0 if k % 3 else 0.8 for k in range(len(inputs))]
    out = []
    for kw in (dict(unfused=True, tail_size=-1), dict(tail_size=-1), dict(tail_size=33), dict()):
        fields = [b.to_field(x) for x in inputs]
        res = lap.solve_batched(fields, dx, 1.0, method="mg_mixed", tol=1e-10, max_iter=3, inner_cycles=inner, **kw)
        torch.cuda.synchronize()
        out.append(([f.cpu().numpy() for f in fields], [(r["iters"], r["r_final"]) for r in res]))
    for got in out[1:]:
        assert got[1] == out[0][1]
        for k in range(len(inputs)):
            assert np.array_equal(got[0][k], out[0][0][k]), SHAPES[k]
    lap.close()


@pytest.mark.parametrize("tiling", [1, 2, 3])
@pytest.mark.parametrize("offset,extra", [(1, 4), (1, 3), (2, 4)])
def test_tiles_update_fields_off_16_byte_boundaries(b, tiling, offset, extra):
    """The tiled level-0 ascent writes psi in pairs of columns: a field that starts 8 bytes past a 16-byte
    boundary, with an even pitch and an odd one, gives what one kernel per pass gives."""
    m, n = 193, 129
    psi = wl.random_ring(m, n, 8)
    lap = b.Laplace()
    outs = []
    for t in (tiling, -1):
        pitch = m + extra + (m + extra) % 2 - (extra % 2)
        buf = torch.zeros(n, pitch, dtype=torch.float64, device="cuda")
        f = buf[:, offset:offset + m]
        f.copy_(torch.as_tensor(psi))
        r = lap.solve(f, method="mg_mixed", tol=1e-10, tiling=t, tail_size=-1)
        outs.append((f.cpu().numpy(), r["iters"], r["status"]))
    lap.close()
    assert outs[0][1:] == outs[1][1:] and outs[0][2] == "converged"
    assert np.array_equal(outs[0][0], outs[1][0])
