"""Workloads of the lattice solver, through its public entry points.

listed() names the cases, draw() makes more of the same ranges, prepare() makes
one's inputs and handles, run() is one pass, work() the bytes and operations a
pass cannot do without, and exact() the same outputs from plain torch in FP64.

Whole solves (hms_solve, hms_solve_batch) are what the library is for, so most
cases are solves: both precisions, uniform and lognormal bars, square and ragged
set grids, set tiles of 16 to 64 nodes, extended relaxation regions, the
twelve-mode form, class factors, several load vectors, host and device memory.
Custom drivers call the single steps; the steps with the most work per node
(residual, update and residual, local relaxation) stand for those.  Solves stop
at R1 < 1e-10 unless the case says otherwise.
"""
import math
import random

import numpy as np
import torch

from paper_1208_4093_gb300 import capi

SQ3 = math.sqrt(3.0)


# ------------------------------------------------------------------ the cases
def _solve(name, nx, ny, sx, sy, **kw):
    c = {"name": name, "kind": "solve", "nx": nx, "ny": ny, "sx": sx, "sy": sy, "ea": "uniform",
         "precision": "fp64", "tol": 1e-10, "nrhs": 1, "overlap": 0, "force": False, "classes": False, "host": False}
    c.update(kw)
    return c


def listed():
    return [
        # a residual check on the smallest lattice a program solves: launch latency
        {"name": "residual_64", "kind": "residual", "nx": 64, "ny": 64, "sx": 16, "sy": 16, "ea": "uniform"},
        # Eq. 3 and the residual on a lattice of 33 M unknowns (mixed form): streaming bandwidth
        {"name": "update_residual_4096_mixed", "kind": "update", "nx": 4096, "ny": 4096, "sx": 64, "sy": 64,
         "ea": "uniform", "precision": "mixed"},
        # a custom driver's relaxation step: 72 sets, ragged last row and column, per-bar stiffness
        {"name": "relax_500x571_fp64", "kind": "relax", "nx": 500, "ny": 571, "sx": 64, "sy": 64, "ea": "lognormal"},
        # the smallest solve: 16 sets, every step latency-bound
        _solve("solve_64_fp64", 64, 64, 16, 16),
        # mid-size lattice of the set-count sweep: 8 x 8 sets of 32 x 32 nodes
        _solve("solve_256_fp64", 256, 256, 32, 32),
        # host buffers in and out, three load cases, sizes no tile divides
        _solve("solve_333x250_mixed_host", 333, 250, 24, 20, ea="lognormal", precision="mixed", nrhs=3, host=True),
        # extended relaxation regions (grown by 4 nodes): few, heavier updates
        _solve("solve_512_overlap4_mixed", 512, 512, 32, 32, ea="lognormal", precision="mixed", overlap=4),
        # the force-controlled modes: twelve per set
        _solve("solve_256x192_force_fp64", 256, 192, 32, 32, ea="lognormal", force=True),
        # the benchmark lattice, plain FP64 form, to the metric's tolerance
        _solve("solve_1024_fp64", 1024, 1024, 64, 64, ea="lognormal", tol=1e-8),
        # the same lattice in the mixed form, to the configuration's tolerance
        _solve("solve_1024_mixed", 1024, 1024, 64, 64, ea="lognormal", precision="mixed"),
        # one factor per class of sets, a set grid too wide for a band factor (35 x 29 sets)
        _solve("solve_1100x900_classes_mixed", 1100, 900, 32, 32, precision="mixed", classes=True),
        # many small uneven lattices at once, one instance per load vector
        {"name": "batch_16_mixed", "kind": "batch", "count": 16, "shapes": 7, "side_min": 32, "side_max": 256,
         "nrhs_max": 4, "precision": "mixed", "tol": 1e-10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _solve_ms(c):
    """A rough time of a solve, to keep drawn cases below the largest listed one."""
    s = max(c["sx"], c["sy"])
    updates = 60 if c["overlap"] >= 2 else (150 if c["overlap"] else 13 * s)
    node = 2.2e-6 if c["precision"] == "fp64" else 1.2e-6
    if c["force"]:
        node *= 2.6
    return c["nrhs"] * updates * (0.35 + node * c["nx"] * c["ny"])


def draw(rng):
    kind = rng.choice(["residual", "update", "relax"] + 6 * ["solve"] + ["batch"])
    while True:
        if kind == "batch":
            return {"kind": kind, "count": rng.randint(4, 16), "shapes": rng.randint(0, 10**6), "side_min": 32,
                    "side_max": rng.randint(96, 256), "nrhs_max": rng.randint(1, 4), "precision": "mixed",
                    "tol": 1e-10}
        ea = rng.choice(["uniform", "lognormal"])
        sx, sy = rng.randint(16, 64), rng.randint(16, 64)
        if rng.random() < 0.5:
            sx = sy = rng.choice([16, 24, 32, 48, 64])
        if kind == "residual":
            return {"kind": kind, "nx": _log(rng, 48, 1024), "ny": _log(rng, 48, 1024), "sx": sx, "sy": sy, "ea": ea}
        if kind == "update":
            sx = sy = rng.choice([32, 48, 64])
            return {"kind": kind, "nx": _log(rng, 256, 4096), "ny": _log(rng, 256, 4096), "sx": sx, "sy": sy,
                    "ea": "uniform", "precision": rng.choice(["fp64", "mixed"])}
        if kind == "relax":
            c = {"kind": kind, "nx": _log(rng, 96, 900), "ny": _log(rng, 96, 900), "sx": sx, "sy": sy, "ea": ea}
            if c["nx"] * c["ny"] <= 600000:
                return c
            continue
        c = _solve("", _log(rng, 48, 800), _log(rng, 48, 800), sx, sy, ea=ea, precision=rng.choice(["fp64", "mixed"]),
                   nrhs=rng.choice([1, 1, 1, 2, 4]), host=rng.random() < 0.3)
        del c["name"]
        form = rng.choice(["plain", "plain", "plain", "overlap", "force", "classes"])
        if form == "overlap":
            c["sx"], c["sy"] = rng.randint(16, 40), rng.randint(16, 40)
            c["overlap"] = rng.randint(1, 8)
        elif form == "force":
            c["force"] = True
        elif form == "classes":
            c["classes"], c["ea"] = True, "uniform"
        # a last row or column of sets one or two nodes wide is not a tiling a program asks for
        if min((c["nx"] - 1) % c["sx"], (c["ny"] - 1) % c["sy"]) < 2:
            continue
        if _solve_ms(c) <= 900.0:
            return c


# ------------------------------------------------------------------ inputs
def _gen(seed, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _device():
    return torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")


def _loads(nrhs, nx, ny, seed, dev):
    """Nodal loads, Uniform(-1, 1) per unknown (the test problem's random loads)."""
    return 2.0 * torch.rand(nrhs, 2 * nx * ny, generator=_gen(4 * seed + 1, dev), device=dev, dtype=torch.float64) - 1.0


def _ea(c, seed, dev):
    """EA per bar [3, ny, nx]: lognormal(0, 0.3), or None for EA = 1 everywhere."""
    if c["ea"] == "uniform":
        return None
    return torch.exp(0.3 * torch.randn(3, c["ny"], c["nx"], generator=_gen(4 * seed + 2, dev), device=dev,
                                       dtype=torch.float64))


def _displacements(nx, ny, seed, dev):
    """A displacement field as a late iterate has it: smooth, with a small rough part."""
    g = _gen(4 * seed + 3, dev)
    x = torch.linspace(0.0, 1.0, nx, device=dev, dtype=torch.float64)
    y = torch.linspace(0.0, 1.0, ny, device=dev, dtype=torch.float64)[:, None]
    u = torch.zeros(ny, nx, 2, device=dev, dtype=torch.float64)
    amp = torch.rand(8, 2, generator=g, device=dev, dtype=torch.float64)
    for k in range(8):
        mode = torch.cos(math.pi * (k % 3) * x) * torch.sin(math.pi * (0.5 + k // 3) * y)
        u += 20.0 * amp[k] * mode[..., None]
    u += 0.1 * torch.randn(ny, nx, 2, generator=g, device=dev, dtype=torch.float64)
    u[0] = 0.0
    return u.reshape(-1).contiguous()


def _step_inputs(c, seed, dev):
    """Displacements, relaxation increment and coefficients of an update: the
    increment is a small part of the displacements, as in the iteration."""
    nx, ny = c["nx"], c["ny"]
    m = -(-nx // c["sx"]) * -(-ny // c["sy"])
    u = _displacements(nx, ny, seed, dev)
    g = _gen(4 * seed + 5, dev)
    delta = 0.01 * torch.randn(ny, nx, 2, generator=g, device=dev, dtype=torch.float64)
    delta[0] = 0.0
    a = torch.randn(m, 9, generator=g, device=dev, dtype=torch.float64)
    size = torch.tensor([1e-2, 1e-2, 1e-4, 1e-4, 1e-4, 1e-4, 1.0, 1e-2, 1e-2], device=dev, dtype=torch.float64)
    return u, delta.reshape(-1).contiguous(), (a * size).reshape(-1).contiguous()


def _batch_shapes(c):
    """(nx, ny, load vectors) of every lattice: long side log-uniform, aspect ratio 1 to 4, either way up."""
    r = random.Random(c["shapes"])
    out = []
    for _ in range(c["count"]):
        a = _log(r, c["side_min"], c["side_max"])
        b = max(8, int(round(a / r.uniform(1.0, 4.0))))
        n = r.randint(1, c["nrhs_max"])
        out.append((a, b, n) if r.random() < 0.5 else (b, a, n))
    return out


def _precision(c):
    return capi.HMS_MIXED if c.get("precision") == "mixed" else capi.HMS_FP64


class _State:
    """What a program keeps between calls: a context, its problems and its buffers."""

    def __init__(self, case):
        self.case = case
        self.ctx = capi.hms_context_create(0)
        self.problems = []

    def problem(self, *args, **kw):
        self.problems.append(capi.hms_problem_create(self.ctx, *args, **kw))
        return self.problems[-1]

    def __del__(self):
        for h in reversed(self.problems):
            capi.hms_problem_destroy(h)
        capi.hms_context_destroy(self.ctx)


def prepare(case, seed):
    c, dev = case, _device()
    s = _State(c)
    f64 = dict(device=dev, dtype=torch.float64)
    if c["kind"] == "batch":
        s.inst, s.loads, s.out = [], [], []
        for k, (nx, ny, nrhs) in enumerate(_batch_shapes(c)):
            # the one-SM upper-level factor for all of them, so that they advance together
            pr = s.problem(nx, ny, 32, 32, precision=_precision(c), tol=c["tol"], max_iter=5000, coarse_factor=4)
            p = _loads(nrhs, nx, ny, 1000 * seed + k, dev)
            for q in range(nrhs):
                if q > 0:
                    s.problems.append(capi.hms_problem_clone(s.ctx, pr))
                s.inst.append(s.problems[-1])
                s.loads.append(p[q:q + 1])
                s.out.append(torch.empty(1, 2 * nx * ny, **f64))
        return s
    nx, ny, nn2 = c["nx"], c["ny"], 2 * c["nx"] * c["ny"]
    ea = _ea(c, seed, dev)
    kw = dict(ea=None if ea is None else ea.cpu().numpy(), precision=_precision(c))
    if c["kind"] == "solve":
        s.pr = s.problem(nx, ny, c["sx"], c["sy"], tol=c["tol"], max_iter=5000, relax_overlap=c["overlap"],
                         mode_mask=0xFFF if c["force"] else 0x1FF, class_factors=int(c["classes"]), **kw)
        s.p = _loads(c["nrhs"], nx, ny, seed, dev)
        s.u = torch.empty(c["nrhs"], nn2, **f64)
        if c["host"]:
            s.p, s.u = s.p.cpu().numpy(), np.empty((c["nrhs"], nn2))
        return s
    s.p = _loads(1, nx, ny, seed, dev)[0]
    if c["kind"] == "relax":
        s.pr = s.problem(nx, ny, c["sx"], c["sy"], **kw)
        s.delta = torch.empty(nn2, **f64)
        s.P = torch.empty(9 * -(-nx // c["sx"]) * -(-ny // c["sy"]), **f64)
        return s
    s.r, s.norms = torch.empty(nn2, **f64), torch.empty(3, **f64)
    if c["kind"] == "residual":
        s.pr = s.problem(nx, ny, c["sx"], c["sy"], **kw)
        s.u = _displacements(nx, ny, seed, dev)
        return s
    # update: the factors are not used by this step; one per class keeps the problem small
    s.pr = s.problem(nx, ny, c["sx"], c["sy"], class_factors=1, **kw)
    s.u, s.delta, s.a = _step_inputs(c, seed, dev)
    s.u_out = torch.empty(nn2, **f64)
    return s


def run(state):
    s, kind = state, state.case["kind"]
    if kind == "solve":
        capi.hms_solve(s.ctx, s.pr, s.p, s.u)
        return s.u
    if kind == "batch":
        capi.hms_solve_batch(s.ctx, s.inst, s.loads, s.out)
        return s.out
    if kind == "relax":
        capi.hms_relax(s.ctx, s.pr, s.p, s.delta, s.P)
        return {"delta": s.delta, "P": s.P}
    if kind == "residual":
        capi.hms_residual(s.ctx, s.pr, s.p, s.u, s.r, s.norms)
        return {"r": s.r, "norms": s.norms}
    capi.hms_update_residual(s.ctx, s.pr, s.p, s.u, s.delta, s.a, s.u_out, s.r, s.norms)
    return {"u": s.u_out, "r": s.r, "norms": s.norms}


def work(case):
    """Per node: p, u, r, delta 16 bytes each, a fixed-DOF byte, 24 bytes of bar
    stiffness where it varies; about 50 operations for the bar forces, 20 for the
    update.  A relaxation solves every set directly, which cannot take fewer
    operations than reading its vectors and one sweep over each bar.  A solve
    reads its loads and writes its displacements; every update in it is a
    relaxation of all sets, an update and a residual."""
    c = case
    if c["kind"] == "batch":
        nodes = sum(nx * ny * n for nx, ny, n in _batch_shapes(c))
        return {"bytes": 32.0 * nodes, "flops": 200.0 * 100 * nodes}
    nodes = c["nx"] * c["ny"]
    bars = 24.0 if c["ea"] == "lognormal" else 0.0
    if c["kind"] == "residual":
        return {"bytes": (49.0 + bars) * nodes, "flops": 50.0 * nodes}
    if c["kind"] == "update":
        return {"bytes": 81.0 * nodes, "flops": 70.0 * nodes}
    if c["kind"] == "relax":
        return {"bytes": (33.0 + bars) * nodes, "flops": 120.0 * nodes}
    updates = 20 if c["overlap"] else 6 * max(c["sx"], c["sy"])
    return {"bytes": c["nrhs"] * (32.0 + bars) * nodes, "flops": c["nrhs"] * updates * 200.0 * nodes}


# ------------------------------------------------------------------ the same in plain FP64
def _bars(nx, ny, ea, dev):
    """EA / L of the E, NE and NW bar of every node, 0 where there is none [3, ny, nx] (L = 1)."""
    k = torch.ones(3, ny, nx, device=dev, dtype=torch.float64) if ea is None else ea.to(dev).clone()
    odd = (torch.arange(ny, device=dev) % 2).bool()
    k[0, :, -1] = 0.0
    k[1:, -1] = 0.0
    k[1, odd, -1] = 0.0   # NE of an odd row goes one column right
    k[2, ~odd, 0] = 0.0   # NW of an even row goes one column left
    return k


def _node_bars(nx, ny, k):
    """For every direction the far node's indices (clipped) and the bar's unit vector."""
    j, i = torch.meshgrid(torch.arange(ny, device=k.device), torch.arange(nx, device=k.device), indexing="ij")
    odd = j % 2
    far = [(i + 1, j), (i + odd, j + 1), (i - 1 + odd, j + 1)]
    e = [(1.0, 0.0), (0.5, 0.5 * SQ3), (-0.5, 0.5 * SQ3)]
    return [(fi.clamp(0, nx - 1), fj.clamp(0, ny - 1), ex, ey) for (fi, fj), (ex, ey) in zip(far, e)]


def _forces(nx, ny, k, u):
    """K u: every bar's axial force on both its nodes."""
    u = u.reshape(ny, nx, 2)
    f = torch.zeros_like(u).reshape(-1, 2)
    own = torch.arange(nx * ny, device=u.device)
    for d, (fi, fj, ex, ey) in enumerate(_node_bars(nx, ny, k)):
        e = torch.tensor([ex, ey], device=u.device, dtype=u.dtype)
        w = u[fj, fi]
        n = (k[d] * ((u - w) @ e))[..., None] * e
        f.index_add_(0, own, n.reshape(-1, 2))
        f.index_add_(0, (fj * nx + fi).reshape(-1), -n.reshape(-1, 2))
    return f.reshape(-1)


def _residual(nx, ny, k, p, u):
    r = (p - _forces(nx, ny, k, u)).reshape(ny, nx, 2).clone()
    r[0] = 0.0
    r = r.reshape(-1)
    pm = p.reshape(ny, nx, 2).clone()
    pm[0] = 0.0
    norms = torch.stack([r.abs().sum(), (r * r).sum(), (u * (pm.reshape(-1) + r)).sum()])
    return r, norms


def _row_blocks(nx, ny, k):
    """Diagonal blocks [ny, 2nx, 2nx] of K row by row and the couplings of row j to row j + 1
    [ny - 1, 2nx, 2nx], the clamped row j = 0 as unit rows."""
    n2, dev = 2 * nx, k.device
    diag = torch.zeros(ny, n2, n2, device=dev, dtype=torch.float64)
    up = torch.zeros(max(ny - 1, 1), n2, n2, device=dev, dtype=torch.float64)  # rows: row j + 1, columns: row j
    j, i = torch.meshgrid(torch.arange(ny, device=dev), torch.arange(nx, device=dev), indexing="ij")
    for d, (fi, fj, ex, ey) in enumerate(_node_bars(nx, ny, k)):
        on = k[d] != 0.0
        jj, ii, fii, fjj, kk = j[on], i[on], fi[on], fj[on], k[d][on]
        e = (ex, ey)
        for a in range(2):
            for b in range(2):
                v = kk * e[a] * e[b]
                diag.index_put_((jj, 2 * ii + a, 2 * ii + b), v, accumulate=True)
                diag.index_put_((fjj, 2 * fii + a, 2 * fii + b), v, accumulate=True)
                if d == 0:
                    diag.index_put_((jj, 2 * ii + a, 2 * fii + b), -v, accumulate=True)
                    diag.index_put_((jj, 2 * fii + a, 2 * ii + b), -v, accumulate=True)
                else:
                    up.index_put_((jj, 2 * fii + a, 2 * ii + b), -v, accumulate=True)
    diag[0] = torch.eye(n2, device=dev, dtype=torch.float64)
    if ny > 1:
        up[0] = 0.0
    return diag, up


def _chain_solve(diag, up, rhs):
    """Block tridiagonal SPD systems, batched: diag(j) [.., m, m], up(j) [.., m, m] the block
    (row j + 1, row j), rhs [.., h, m, q]."""
    h = rhs.shape[-3]
    inv, y = [], []
    for j in range(h):
        d, b = diag(j), rhs[..., j, :, :]
        if j > 0:
            t = up(j - 1)
            g = torch.cholesky_solve(t.transpose(-1, -2).contiguous(), inv[-1])
            d, b = d - t @ g, b - g.transpose(-1, -2) @ y[-1]
        inv.append(torch.linalg.cholesky(d))
        y.append(b)
    x = [None] * h
    for j in range(h - 1, -1, -1):
        b = y[j] if j + 1 == h else y[j] - up(j).transpose(-1, -2) @ x[j + 1]
        x[j] = torch.cholesky_solve(b, inv[j])
    return torch.stack(x, dim=-3)


def _direct(nx, ny, ea, p, dev):
    """u = K^-1 p over the free unknowns; None where plain torch would take too long."""
    if (2.0 * nx) ** 3 * ny > 1.2e12 or (2.0 * nx) ** 2 * ny * 8 > 8e9:
        return None
    diag, up = _row_blocks(nx, ny, _bars(nx, ny, ea, dev))
    b = p.reshape(-1, ny, 2 * nx).permute(1, 2, 0).clone()
    b[0] = 0.0
    x = _chain_solve(lambda j: diag[j], lambda j: up[j], b)
    return x.permute(2, 0, 1).reshape(p.shape)


def _centroids(c, dev):
    """xi and eta of every node against its set's centroid, and its set [ny, nx]."""
    nx, ny, sx, sy = c["nx"], c["ny"], c["sx"], c["sy"]
    j, i = torch.meshgrid(torch.arange(ny, device=dev), torch.arange(nx, device=dev), indexing="ij")
    mx, my = -(-nx // sx), -(-ny // sy)
    own = (j // sy) * mx + i // sx
    x, y = i + 0.5 * (j % 2).double(), 0.5 * SQ3 * j.double()
    one = torch.ones_like(x)
    total = [torch.zeros(mx * my, device=dev, dtype=torch.float64).index_add_(0, own.reshape(-1), v.reshape(-1).double())
             for v in (one, x, y)]
    return x - (total[1] / total[0])[own], y - (total[2] / total[0])[own], own


def _relax(c, k, r):
    """Every set's k^Inner^-1 r_I, and V^T r of the nine modes built from it."""
    nx, ny, sx, sy, dev = c["nx"], c["ny"], c["sx"], c["sy"], r.device
    r = r.reshape(ny, nx, 2).clone()
    r[0] = 0.0
    delta = torch.zeros_like(r)
    # the rows' blocks are cut set column by set column: [ny, 2w, 2w] of each
    for i0 in range(0, nx, sx):
        w = min(sx, nx - i0)
        sub = torch.zeros(3, ny, nx, device=dev, dtype=torch.float64)
        lo, hi = max(i0 - 1, 0), min(i0 + w + 1, nx)
        sub[:, :, lo:hi] = k[:, :, lo:hi]
        a, cut = max(i0 - 2, 0), min(i0 + w + 2, nx)
        diag, up = _row_blocks(cut - a, ny, sub[:, :, a:cut].contiguous())
        m = slice(2 * (i0 - a), 2 * (i0 - a + w))
        diag, up = diag[:, m, m], up[:, m, m]
        for h in sorted({min(sy, ny - j0) for j0 in range(0, ny, sy)}):
            rows = [j0 for j0 in range(0, ny, sy) if min(sy, ny - j0) == h]
            at = torch.tensor(rows, device=dev)
            b = torch.stack([r[j0:j0 + h, i0:i0 + w].reshape(h, 2 * w, 1) for j0 in rows])
            x = _chain_solve(lambda j: diag[at + j], lambda j: up[at + j], b)
            for q, j0 in enumerate(rows):
                delta[j0:j0 + h, i0:i0 + w] = x[q].reshape(h, w, 2)
    xi, eta, own = _centroids(c, dev)
    dr = (delta * r).sum(-1)
    v = torch.stack([r[..., 0], r[..., 1], xi * r[..., 0], eta * r[..., 0], xi * r[..., 1], eta * r[..., 1], dr,
                     xi * dr, eta * dr], dim=-1)
    m = -(-nx // sx) * -(-ny // sy)
    P = torch.zeros(m, 9, device=dev, dtype=torch.float64).index_add_(0, own.reshape(-1), v.reshape(-1, 9))
    return delta.reshape(-1), P.reshape(-1)


def _updated(c, u, delta, a):
    """u + V a with the nine modes of every set (0 on the clamped row)."""
    nx, ny = c["nx"], c["ny"]
    xi, eta, own = _centroids(c, u.device)
    q = a.reshape(-1, 9)[own]
    d = delta.reshape(ny, nx, 2)
    cd = q[..., 6] + q[..., 7] * xi + q[..., 8] * eta
    inc = torch.stack([q[..., 0] + q[..., 2] * xi + q[..., 3] * eta + cd * d[..., 0],
                       q[..., 1] + q[..., 4] * xi + q[..., 5] * eta + cd * d[..., 1]], dim=-1)
    inc[0] = 0.0
    return u + inc.reshape(-1)


def exact(case, seed):
    c, dev = case, _device()
    if c["kind"] == "batch":
        out = []
        for k, (nx, ny, nrhs) in enumerate(_batch_shapes(c)):
            u = _direct(nx, ny, None, _loads(nrhs, nx, ny, 1000 * seed + k, dev), dev)
            out += [u[q:q + 1] for q in range(nrhs)]
        return out
    nx, ny, ea = c["nx"], c["ny"], _ea(c, seed, dev)
    if c["kind"] == "solve":
        u = _direct(nx, ny, ea, _loads(c["nrhs"], nx, ny, seed, dev), dev)
        return u.cpu().numpy() if u is not None and c["host"] else u
    k, p = _bars(nx, ny, ea, dev), _loads(1, nx, ny, seed, dev)[0]
    if c["kind"] == "relax":
        delta, P = _relax(c, k, p)
        return {"delta": delta, "P": P}
    if c["kind"] == "residual":
        r, norms = _residual(nx, ny, k, p, _displacements(nx, ny, seed, dev))
        return {"r": r, "norms": norms}
    u = _updated(c, *_step_inputs(c, seed, dev))
    r, norms = _residual(nx, ny, k, p, u)
    return {"u": u, "r": r, "norms": norms}
