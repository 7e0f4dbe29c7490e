"""The update and residual (Eqs. 3, 1) where the kernel's layout changes: warps
of 30 columns and a size-dependent count of rows (one on small lattices, more
on large ones), sets of a few nodes and larger ones, a set's edge inside a
warp's rows and columns.

u + V a against the modes' definition (1e-13 in FP64; in the mixed form the
increment's FP32 rounding, 2e-6 of its largest term, except for sets of a few
nodes, whose increment is FP64 on an FP32 delta); r against the oracle's
residual of the u returned (1e-12 of the loads and bar forces).
"""
import numpy as np
import pytest

from oracle import hms, truss
from workloads import ea_lognormal, loads

pytestmark = pytest.mark.gpu

# nx, ny, sx, sy, lognormal EA
CASES = [(2, 2, 2, 2, True), (30, 5, 7, 3, False), (31, 33, 31, 33, True), (61, 47, 9, 4, True), (59, 64, 3, 3, False),
         (300, 260, 64, 64, True), (420, 700, 20, 33, False)]


def increment(tr, g, d, a):
    """V a and the sum of its terms' sizes, in extended precision: the oracle's
    own doubles carry the rounding of coordinates of several hundred bars, up to
    the tolerance here.  The representing points are those doubles the library
    takes (the centroid of a set's nodes)."""
    X = np.longdouble
    nx, ny, sx, sy = tr.nx, tr.ny, g.sx, g.sy
    hh = 0.86602540378443864676
    j, i = np.divmod(np.arange(nx * ny), nx)
    Ix, Iy = i // sx, j // sy
    i0, j0 = np.arange(g.Mx) * sx, np.arange(g.My) * sy
    w, h = np.minimum(sx, nx - i0), np.minimum(sy, ny - j0)
    odd = (j0 + h) // 2 - j0 // 2
    cx = (i0 + 0.5 * (w - 1))[None, :] + 0.5 * (odd / h)[:, None]
    cy = hh * (j0 + 0.5 * (h - 1))
    xi = i + X(0.5) * (j % 2) - cx[Iy, Ix].astype(X)
    eta = X(hh) * j - cy[Iy].astype(X)
    A = a.reshape(-1, 9)[Iy * g.Mx + Ix].astype(X)
    D = d.reshape(-1, 2).astype(X)
    out, size = np.empty((nx * ny, 2), X), np.empty((nx * ny, 2), X)
    for f in (0, 1):
        t = [A[:, f], A[:, 2 + 2 * f] * xi, A[:, 3 + 2 * f] * eta, A[:, 6] * D[:, f], A[:, 7] * xi * D[:, f],
             A[:, 8] * eta * D[:, f]]
        out[:, f], size[:, f] = sum(t), sum(np.abs(q) for q in t)
    return out.reshape(-1) * tr.free, size.reshape(-1)


@pytest.mark.parametrize("case", CASES, ids=["x".join(map(str, c[:4])) for c in CASES])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_update_residual(hms_ctx, case, prec):
    from paper_1208_4093_gb300 import capi
    nx, ny, sx, sy, ln = case
    ea = ea_lognormal(nx, ny, 3) if ln else None
    tr = truss.Truss(nx, ny, ea)
    g = hms.SetGrid(nx, ny, sx, sy)
    rng = np.random.default_rng(nx + ny)
    p = tr.free * loads(nx, ny, 2).reshape(-1)
    u = tr.free * rng.standard_normal(tr.ndof)
    d = (tr.free * rng.standard_normal(tr.ndof)).astype(np.float32).astype(np.float64)
    a = rng.standard_normal(9 * g.M)
    pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, ea=ea, precision=prec, class_factors=int(not ln))
    try:
        uo, ro, nrm = np.empty(tr.ndof), np.empty(tr.ndof), np.empty(3)
        capi.hms_update_residual(hms_ctx, pr, p, u, d, a, uo, ro, nrm)
        r0, n0 = np.empty(tr.ndof), np.empty(3)
        capi.hms_residual(hms_ctx, pr, p, uo, r0, n0)
    finally:
        capi.hms_problem_destroy(pr)
    inc, scale = increment(tr, g, d, a)
    assert np.all(np.abs(uo - (u + inc)) <= (2e-6 if prec else 1e-13) * (scale + np.abs(u)))
    assert np.all(uo[~tr.free] == 0)
    want = tr.residual(p, uo)
    size = np.linalg.norm(p) + np.linalg.norm(want - p)
    assert np.linalg.norm(ro - want) < 1e-12 * size
    # the residual of the returned u: the same bits, with and without the update
    assert np.array_equal(r0, ro) and np.array_equal(n0, nrm)
    ref = [np.abs(ro).sum(), ro @ ro, uo @ (p + ro)]
    assert np.allclose(nrm[:2], ref[:2], rtol=1e-12) and abs(nrm[2] - ref[2]) < 1e-12 * np.abs(uo) @ np.abs(p + ro)


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("mask", [0x1FF, 0xFFF])
def test_update_residual_device_buffers(hms_ctx, prec, mask):
    """Device buffers used in place, buffers that start off a 16-byte boundary
    and outputs that overlap inputs (both through the problem's own buffers)
    give the bits of the host call."""
    torch = pytest.importorskip("torch")
    from paper_1208_4093_gb300 import capi
    nx, ny, sx, sy = 50, 42, 24, 20
    tr = truss.Truss(nx, ny)
    g = hms.SetGrid(nx, ny, sx, sy)
    q = 12 if mask == 0xFFF else 9
    rng = np.random.default_rng(1)
    # u not zero on constrained DOFs: it is read as zero there
    p, u = rng.standard_normal(tr.ndof), rng.standard_normal(tr.ndof)
    d, a = rng.standard_normal(tr.ndof * (2 if q == 12 else 1)), rng.standard_normal(q * g.M)
    pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, precision=prec, mode_mask=mask)
    try:
        host = [np.empty(tr.ndof), np.empty(tr.ndof), np.empty(3)]
        capi.hms_update_residual(hms_ctx, pr, p, u, d, a, *host)
        for off in (0, 1):
            def dev(x):
                t = torch.empty(x.size + off, dtype=torch.float64, device="cuda")[off:]
                t.copy_(torch.from_numpy(x))
                return t
            P, U, D, A = dev(p), dev(u), dev(d), dev(a)
            outs = [dev(np.zeros(tr.ndof)), dev(np.zeros(tr.ndof)), dev(np.zeros(3))]
            torch.cuda.synchronize()
            capi.hms_update_residual(hms_ctx, pr, P, U, D, A, *outs)
            for h, o in zip(host, outs):
                assert np.array_equal(h, o.cpu().numpy())
            assert np.array_equal(U.cpu().numpy(), u) and np.array_equal(P.cpu().numpy(), p)
            capi.hms_update_residual(hms_ctx, pr, P, U, D, A, U, P, outs[2])  # u and p overwritten
            assert np.array_equal(host[0], U.cpu().numpy()) and np.array_equal(host[1], P.cpu().numpy())
            assert np.array_equal(host[2], outs[2].cpu().numpy())
    finally:
        capi.hms_problem_destroy(pr)
