"""The work that users of this library have it do, as cases that can be timed and compared.

A case is a dict of plain values; listed() names the standing ones and draw() gives others of
the same ranges. prepare() makes the inputs (on the device, from a seed) and the handle that a
program keeps; run() is one pass through the public entry points of binding.py; exact() is the
same result in plain 64-bit torch.

Every solve starts from freshly copied data (a boundary ring and a zero interior), as a program
does when new boundary values arrive in the field it keeps.
"""
import math

import torch

from paper_2208_02427_gb300 import binding as b
from paper_2208_02427_gb300 import workloads as wl


def listed():
    return [
        # The paper's own problem (25 x 17, stop at max |change| <= 1e-9) by point SOR at its
        # optimum: the smallest call, all latency.
        {"name": "chamber_sor", "kind": "small", "method": "sor", "m": 25, "n": 17, "w": 1.75},
        # The same problem by zebra ADI, form B, at its optimum: the smallest line solve.
        {"name": "chamber_adi", "kind": "small", "method": "adi", "m": 25, "n": 17, "w": 1.3},
        # An everyday SOR solve to 1e-10 on a ragged grid that fits in cache: thousands of short
        # launches.
        {"name": "sor_513x385", "kind": "point", "method": "sor", "m": 513, "n": 385, "order": "paper",
         "sweeps": 3000, "every": 100, "tol": 1e-10, "aspect": 1.0},
        # Two check periods of the full-size SOR solve (neighbour sums paired along diagonals).
        {"name": "sor_4097", "kind": "point", "method": "sor", "m": 4097, "n": 4097, "order": "diagonal",
         "sweeps": 200, "every": 100, "tol": 0.0, "aspect": 1.0},
        # Jacobi sweeps on a ragged grid of medium size.
        {"name": "jacobi_1531x1021", "kind": "point", "method": "jacobi", "m": 1531, "n": 1021,
         "order": "paper", "sweeps": 100, "every": 50, "tol": 0.0, "aspect": 1.0},
        # ADI iterations on a large ragged grid with dx != dy: both line directions.
        {"name": "adi_3001x2050", "kind": "line", "method": "adi", "form": "A", "m": 3001, "n": 2050,
         "w": 1.3, "iters": 10, "aspect": 1.25},
        # A small FP64 multigrid solve: latency of the coarse levels.
        {"name": "mg_257x129", "kind": "mg", "method": "mg", "m": 257, "n": 129, "aspect": 1.0},
        # The full-size FP64 multigrid solve.
        {"name": "mg_4097", "kind": "mg", "method": "mg", "m": 4097, "n": 4097, "aspect": 1.0},
        # An ordinary mixed-precision solve, sides not powers of two.
        {"name": "mixed_1537x1025", "kind": "mg", "method": "mg_mixed", "m": 1537, "n": 1025, "aspect": 1.0},
        # The largest mixed-precision solve.
        {"name": "mixed_8193", "kind": "mg", "method": "mg_mixed", "m": 8193, "n": 8193, "aspect": 1.0},
        # A thousand uneven grids solved together.
        {"name": "batch_mixed_1024", "kind": "batch", "method": "mg_mixed", "count": 1024, "kmin": 5,
         "kmax": 9, "shapes": 3},
        # A burst of requests through the server: multigrid and SOR of many sizes sharing steps.
        {"name": "serve_48", "kind": "serve", "count": 48, "kmin": 5, "kmax": 10, "shapes": 7},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mg_side(rng, lo, hi):
    """A side (2, 3, 5 or 7) 2^k + 1 in [lo, hi]."""
    sides = [f * 2 ** k + 1 for f in (2, 2, 3, 5, 7) for k in range(2, 13) if lo <= f * 2 ** k + 1 <= hi]
    want = _log_int(rng, lo, hi)
    near = sorted(sides, key=lambda s: abs(math.log(s / want)))[:3]
    return rng.choice(near)


def _mg_case(rng):
    while True:
        m = _mg_side(rng, 33, 6145)
        n = _mg_side(rng, max(33, m // 4), min(6145, 4 * m))
        mc, nc = _levels(m, n)[-1]
        # the coarsest level is solved directly and stays small on sides worth coarsening
        if (mc - 2) * (nc - 2) <= 256:
            return {"kind": "mg", "method": rng.choice(["mg", "mg_mixed"]), "m": m, "n": n,
                    "aspect": rng.choice([1.0, 1.0, 1.0, 0.8, 1.25])}


def draw(rng):
    kind = rng.choice(["small", "point", "point", "line", "mg", "mg", "mg", "batch", "batch", "serve"])
    if kind == "small":
        method = rng.choice(["sor", "sor", "adi", "slor", "jacobi"])
        m, n = rng.randint(9, 61), rng.randint(9, 61)
        w = {"sor": round(wl.w_opt_sor(m, n), 3), "adi": 1.3, "slor": 1.25, "jacobi": 1.0}[method]
        return {"kind": "small", "method": method, "m": m, "n": n, "w": w}
    if kind == "point":
        m = _log_int(rng, 65, 4096)
        n = _log_int(rng, max(65, m // 4), min(4096, 4 * m))
        method = rng.choice(["sor", "sor", "gs", "jacobi"])
        order = rng.choice(["paper", "diagonal"]) if method != "jacobi" else "paper"
        aspect = 1.0 if order == "diagonal" else rng.choice([1.0, 1.0, 0.8])
        return {"kind": "point", "method": method, "m": m, "n": n, "order": order, "sweeps": 200,
                "every": rng.choice([20, 50, 100]), "tol": 0.0, "aspect": aspect}
    if kind == "line":
        m, n = _log_int(rng, 129, 4096), _log_int(rng, 129, 4096)
        return {"kind": "line", "method": rng.choice(["adi", "slor"]), "form": rng.choice(["A", "B"]),
                "m": m, "n": n, "w": round(rng.uniform(1.0, 1.35), 3), "iters": 10,
                "aspect": rng.choice([1.0, 1.25])}
    if kind == "mg":
        return _mg_case(rng)
    if kind == "batch":
        return {"kind": "batch", "method": rng.choice(["mg", "mg_mixed"]), "count": _log_int(rng, 24, 1024),
                "kmin": 5, "kmax": rng.choice([8, 9]), "shapes": rng.randrange(1, 1000)}
    return {"kind": "serve", "count": _log_int(rng, 8, 48), "kmin": 5, "kmax": 9,
            "shapes": rng.randrange(1, 1000)}


# ---- inputs ----------------------------------------------------------------------------

def _ring(psi, seed):
    """Each edge of psi (n, m) a sum of eight sine modes with U[-1, 1] coefficients; corners and
    interior 0 (the recipe of workloads.sine_edges, made on the device)."""
    n, m = psi.shape
    a = torch.as_tensor(wl.sine_coefficients(seed)).to(psi.device)
    k = math.pi * torch.arange(1, a.shape[1] + 1, device=psi.device, dtype=torch.float64)[:, None]
    sx = torch.sin(k * torch.linspace(0, 1, m, device=psi.device, dtype=torch.float64))
    sy = torch.sin(k * torch.linspace(0, 1, n, device=psi.device, dtype=torch.float64))
    psi.zero_()
    psi[0], psi[-1] = a[0] @ sx, a[1] @ sx
    psi[1:-1, 0], psi[1:-1, -1] = (a[2] @ sy)[1:-1], (a[3] @ sy)[1:-1]
    psi[0, 0] = psi[0, -1] = psi[-1, 0] = psi[-1, -1] = 0.0


def _spacing(case):
    dx = 1.0 / (case["m"] - 1)
    return dx, dx * case["aspect"]


def _shapes(case):
    return wl.batch_shapes(case["count"], seed=case["shapes"], kmin=case["kmin"], kmax=case["kmax"])


def _many(shapes, seed):
    """Fields of the given (m, n) in one buffer, U[0, 1] rings and zero interiors: the buffer, its
    views, and the index of every ring entry."""
    offs, views, total = [], [], 0
    for m, n in shapes:
        pitch = (m + 31) // 32 * 32
        offs.append((total, m, n, pitch))
        total += n * pitch
    buf = torch.zeros(total, dtype=torch.float64, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(seed)
    noise = torch.rand(sum(2 * m + 2 * n for m, n in shapes), generator=g, dtype=torch.float64, device="cuda")
    at = 0
    for off, m, n, pitch in offs:
        v = buf[off:off + n * pitch].view(n, pitch)[:, :m]
        v[0] = noise[at:at + m]
        v[-1] = noise[at + m:at + 2 * m]
        v[1:-1, 0] = noise[at + 2 * m:at + 2 * m + n - 2]
        v[1:-1, -1] = noise[at + 2 * m + n:at + 2 * m + 2 * n - 2]
        at += 2 * m + 2 * n
        views.append(v)
    return buf, views


def prepare(case, seed):
    lap = b.Laplace()
    s = {"case": case, "lap": lap}
    if case["kind"] in ("batch", "serve"):
        s["start"], _ = _many(_shapes(case), seed)
        s["buf"], s["fields"] = s["start"].clone(), None
        at, fields = 0, []
        for m, n in _shapes(case):
            pitch = (m + 31) // 32 * 32
            fields.append(s["buf"][at:at + n * pitch].view(n, pitch)[:, :m])
            at += n * pitch
        s["fields"] = fields
        if case["kind"] == "batch":
            s["batch"] = b.Batch(fields)
        else:
            s["server"] = b.Server(lap, hbm_budget=4 << 30)
            s["asks"] = _requests(case)
        return s
    m, n = case["m"], case["n"]
    s["start"], s["psi"] = b.field(m, n), b.field(m, n)
    if case["kind"] == "small":
        # the chamber: one wall at a constant value near 1, the others at 0
        g = torch.Generator().manual_seed(seed)
        s["start"][0, 1:m - 1] = 0.75 + 0.5 * torch.rand(1, generator=g, dtype=torch.float64).item()
    else:
        _ring(s["start"], seed)
    s["psi"].copy_(s["start"])
    return s


def _requests(case):
    """Method, w, tolerance of each request: half mixed multigrid, half SOR, tolerances 1e-6 ..
    1e-9 in turn."""
    out = []
    for k, (m, n) in enumerate(_shapes(case)):
        sor = k % 2 == 1
        out.append({"method": "sor" if sor else "mg_mixed", "w": wl.w_opt_sor(m, n) if sor else 1.0,
                    "tol": 10.0 ** -(6 + k // 2 % 4)})
    return out


# ---- one pass ----------------------------------------------------------------------------

_STATUS = {v: k for k, v in b.STATUS.items()}


def run(s):
    # iteration counts come back with the field; the norms reported beside them are the stopping
    # test's own (about six digits in the mixed solver) and stay out
    case, lap = s["case"], s["lap"]
    kind = case["kind"]
    if kind == "batch":
        s["buf"].copy_(s["start"])
        res = lap.solve_batched(s["batch"], method=case["method"], tol=1e-10, max_iter=100)
        return {"psi": s["buf"], "iters": torch.tensor([r["iters"] for r in res]),
                "status": torch.tensor([_STATUS[r["status"]] for r in res])}
    if kind == "serve":
        s["buf"].copy_(s["start"])
        srv = s["server"]
        ids = [srv.submit(f, **a) for f, a in zip(s["fields"], s["asks"])]
        while sum(srv.step()):
            pass
        res = dict(srv.drain())
        return {"psi": s["buf"], "iters": torch.tensor([res[i]["iters"] for i in ids]),
                "status": torch.tensor([_STATUS[res[i]["status"]] for i in ids])}
    psi = s["psi"]
    psi.copy_(s["start"])
    if kind == "small":
        r = lap.solve(psi, 0.25, 0.25, method=case["method"], w=case["w"], tol=1e-9, norm="maxdelta",
                      max_iter=20000, line_form="B")
    elif kind == "point":
        r = lap.solve(psi, *_spacing(case), method=case["method"], w=_point_w(case), tol=case["tol"],
                      max_iter=case["sweeps"], check_every=case["every"], sum_order=case["order"])
    elif kind == "line":
        r = lap.solve(psi, *_spacing(case), method=case["method"], w=case["w"], tol=0.0,
                      max_iter=case["iters"], check_every=case["iters"], line_form=case["form"])
    else:
        r = lap.solve(psi, *_spacing(case), method=case["method"], tol=1e-10, max_iter=100)
    return {"psi": psi, "iters": r["iters"], "status": _STATUS[r["status"]]}


def _point_w(case):
    if case["method"] != "sor":
        return 1.0
    return wl.w_opt_sor(case["m"], case["n"], 1.0 / case["aspect"])


# ---- what a pass cannot do without --------------------------------------------------------

def work(case):
    """Bytes: every field read and written once. Flops: the method's floating-point operations per
    interior point times its iterations (about what the tolerance takes where it is not fixed)."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        shapes = _shapes(case)
        points = sum(m * n for m, n in shapes)
        if kind == "batch":
            return {"bytes": 16.0 * points, "flops": 8 * 34.0 * points}
        flops = sum(m * n * (5.0 * 2.2 * max(m, n) if k % 2 else 8 * 34.0) for k, (m, n) in enumerate(shapes))
        return {"bytes": 16.0 * points, "flops": flops}
    points = case["m"] * case["n"]
    if kind == "small":
        rate = {"sor": (5.0, 3.5), "adi": (16.0, 4.0), "slor": (8.0, 3.0), "jacobi": (4.0, 50.0)}[case["method"]]
        flops = rate[0] * rate[1] * max(case["m"], case["n"]) * points
    elif kind == "point":
        sweeps = case["sweeps"] if case["tol"] == 0.0 else 2.7 * max(case["m"], case["n"])
        flops = {"sor": 6.0, "gs": 4.0, "jacobi": 4.0}[case["method"]] * sweeps * points
    elif kind == "line":
        flops = (8.0 if case["method"] == "slor" else 16.0) * case["iters"] * points
    else:
        flops = 7 * 34.0 * points
    return {"bytes": 16.0 * points, "flops": flops}


# ---- the same results in plain 64-bit torch ------------------------------------------------

def _sum4(u, b2):
    return (u[..., 1:-1, 2:] + u[..., 1:-1, :-2]) + b2 * (u[..., 2:, 1:-1] + u[..., :-2, 1:-1])


def _parity(n, m, device):
    j = torch.arange(1, n - 1, device=device)[:, None]
    i = torch.arange(1, m - 1, device=device)[None, :]
    return (i + j) % 2


def _rb_sweep(u, q, b2, w, red):
    """One red-black sweep in place; red: the boolean masks of the red and the black points."""
    inner = u[..., 1:-1, 1:-1]
    for mask in red:
        s = _sum4(u, b2)
        if q is not None:
            s += q[..., 1:-1, 1:-1]
        s *= w / (2.0 * (1.0 + b2))
        if w != 1.0:
            s += (1.0 - w) * inner
        inner.copy_(torch.where(mask, s, inner))


def _masks(u):
    p = _parity(u.shape[-2], u.shape[-1], u.device)
    return p == 0, p == 1


def _defect(u, q, b2):
    r = torch.zeros_like(u)
    r[..., 1:-1, 1:-1] = _sum4(u, b2) - 2.0 * (1.0 + b2) * u[..., 1:-1, 1:-1]
    if q is not None:
        r[..., 1:-1, 1:-1] += q[..., 1:-1, 1:-1]
    return r


def _levels(m, n):
    out = [(m, n)]
    while (m - 1) % 2 == 0 and (n - 1) % 2 == 0 and min((m - 1) // 2, (n - 1) // 2) + 1 >= 5:
        m, n = (m - 1) // 2 + 1, (n - 1) // 2 + 1
        out.append((m, n))
    return out


def _second_difference(k, device):
    e = torch.ones(k - 1, dtype=torch.float64, device=device)
    return torch.diag(e, 1) + torch.diag(e, -1) - 2.0 * torch.eye(k, dtype=torch.float64, device=device)


def _vcycle(u, q, b2, depth):
    if depth == 0:
        m, n = u.shape[-1] - 2, u.shape[-2] - 2
        eye = lambda k: torch.eye(k, dtype=torch.float64, device=u.device)  # noqa: E731
        A = (torch.kron(eye(n), _second_difference(m, u.device)) +
             b2 * torch.kron(_second_difference(n, u.device), eye(m)))
        r = _defect(u, q, b2)[..., 1:-1, 1:-1].reshape(u.shape[0], -1)
        u[..., 1:-1, 1:-1] -= torch.linalg.solve(A, r.T).T.reshape(-1, n, m)
        return
    masks = _masks(u)
    for _ in range(2):
        _rb_sweep(u, q, b2, 1.0, masks)
    r = _defect(u, q, b2)
    fw = torch.zeros_like(r[..., ::2, ::2])
    c = r[..., 2:-2:2, 2:-2:2]
    edges = r[..., 2:-2:2, 1:-3:2] + r[..., 2:-2:2, 3:-1:2] + r[..., 1:-3:2, 2:-2:2] + r[..., 3:-1:2, 2:-2:2]
    corners = (r[..., 1:-3:2, 1:-3:2] + r[..., 1:-3:2, 3:-1:2] + r[..., 3:-1:2, 1:-3:2] + r[..., 3:-1:2, 3:-1:2])
    fw[..., 1:-1, 1:-1] = 0.25 * (4.0 * c + 2.0 * edges + corners)
    e = torch.zeros_like(fw)
    _vcycle(e, fw, b2, depth - 1)
    rows = torch.zeros(u.shape[:-1] + (e.shape[-1],), dtype=u.dtype, device=u.device)
    rows[..., ::2, :] = e
    rows[..., 1::2, :] = 0.5 * (e[..., 1:, :] + e[..., :-1, :])
    u[..., ::2] += rows
    u[..., 1::2] += 0.5 * (rows[..., 1:] + rows[..., :-1])
    for _ in range(2):
        _rb_sweep(u, q, b2, 1.0, masks)


def _norms(u, b2):
    return _defect(u, None, b2).flatten(1).norm(dim=1)


def _mg_solve(u, b2):
    """V(2,2) cycles on the stack u (k, n, m), each field until its residual is 1e-10 of its first."""
    depth = len(_levels(u.shape[-1], u.shape[-2])) - 1
    r0 = _norms(u, b2)
    for _ in range(100):
        on = _norms(u, b2) > 1e-10 * r0
        if not bool(on.any()):
            break
        v = u[on]
        _vcycle(v, None, b2, depth)
        u[on] = v
    return u


def _line_sweep(u, w, b2, form, direction):
    """Zebra line relaxation: odd lines, then even ones, each line solved exactly."""
    if direction == 1:
        u, off, cross = u.T, b2, 1.0
    else:
        off, cross = 1.0, b2
    d, k = 2.0 * (1.0 + b2), u.shape[1] - 2
    a = off if form == "A" else w * off
    e = torch.full((k - 1,), -a, dtype=u.dtype, device=u.device)
    T = torch.diag(e, 1) + torch.diag(e, -1) + d * torch.eye(k, dtype=u.dtype, device=u.device)
    inv = torch.linalg.inv(T)
    for first in (1, 2):
        line = u[first:-1:2]
        rhs = cross * (u[first - 1:-2:2] + u[first + 1::2])[:, 1:-1]
        if form == "B":
            rhs = w * rhs + d * (1.0 - w) * line[:, 1:-1]
        rhs[:, 0] += a * line[:, 0]
        rhs[:, -1] += a * line[:, -1]
        x = rhs @ inv  # T is symmetric
        line[:, 1:-1] = x if form == "B" else w * x + (1.0 - w) * line[:, 1:-1]


def _jacobi_sweep(u, b2):
    u[1:-1, 1:-1] = _sum4(u, b2) / (2.0 * (1.0 + b2))


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return None  # thousands of sweeps of dozens of grids: minutes in plain torch
    if kind == "batch":
        buf, views = _many(_shapes(case), seed)
        groups = {}
        for v in views:
            groups.setdefault(tuple(v.shape), []).append(v)
        for vs in groups.values():
            for v, x in zip(vs, _mg_solve(torch.stack(vs), 1.0)):
                v.copy_(x)
        return {"psi": buf, "iters": None, "status": None}
    u = torch.zeros(case["n"], case["m"], dtype=torch.float64, device="cuda")
    if kind == "small":
        g = torch.Generator().manual_seed(seed)
        u[0, 1:-1] = 0.75 + 0.5 * torch.rand(1, generator=g, dtype=torch.float64).item()
        b2, masks = 1.0, _masks(u)
        for _ in range(20000):
            old = u.clone()
            if case["method"] == "sor":
                _rb_sweep(u, None, b2, case["w"], masks)
            elif case["method"] == "jacobi":
                _jacobi_sweep(u, b2)
            else:
                _line_sweep(u, case["w"], b2, "B", 0)
                if case["method"] == "adi":
                    _line_sweep(u, case["w"], b2, "B", 1)
            if (u - old).abs().max().item() <= 1e-9:
                break
        return {"psi": u, "iters": None, "status": None}
    _ring(u, seed)
    dx, dy = _spacing(case)
    b2 = (dx / dy) ** 2
    if kind == "mg":
        return {"psi": _mg_solve(u[None], b2)[0], "iters": None, "status": None}
    if kind == "line":
        for _ in range(case["iters"]):
            _line_sweep(u, case["w"], b2, case["form"], 0)
            if case["method"] == "adi":
                _line_sweep(u, case["w"], b2, case["form"], 1)
        return {"psi": u, "iters": None, "status": None}
    masks, r0, w = _masks(u), _norms(u[None], b2), _point_w(case)
    for k in range(1, case["sweeps"] + 1):
        if case["method"] == "jacobi":
            _jacobi_sweep(u, b2)
        else:
            _rb_sweep(u, None, b2, w, masks)
        if k % case["every"] == 0 and bool(_norms(u[None], b2) <= case["tol"] * r0):
            break
    return {"psi": u, "iters": None, "status": None}
