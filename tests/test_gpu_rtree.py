"""The relaxation by nested dissection of every set (relax_tree.cu) at the tile
sizes where its plan changes: just above the 64 nodes from which it runs, one
and two nodes wide, fronts of one and several 32-unknown panels, boxes cut once
or twice, ragged last sets, up to the 64 x 64 nodes of the largest tile, grown
regions, fixed DOFs inside sets, and the cut-free factors (Eq. 15).

delta (Eq. 13) against the oracle's per-set local solves (Eq. 12) at the
tolerances of test_gpu_parity: FP64 1e-11, FP32 2e-5; P (Eq. 7) against the
modes of that delta.  CTA sizes must agree bit for bit.
"""
import numpy as np
import pytest

from oracle import hms, truss
from workloads import ea_lognormal, loads

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(np.asarray(a) - b) / np.linalg.norm(b)


# nx, ny, sx, sy, overlap
CASES = [(20, 17, 9, 8, 0), (27, 14, 13, 5, 0), (70, 3, 64, 2, 0), (3, 150, 1, 80, 0), (5, 140, 2, 65, 0),
         (40, 40, 17, 16, 0), (50, 41, 24, 20, 0), (64, 64, 64, 64, 0), (65, 63, 33, 62, 0), (48, 40, 16, 9, 3),
         (75, 30, 12, 12, 8)]


@pytest.mark.parametrize("case", CASES, ids=["x".join(map(str, c)) for c in CASES])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_relax_step(hms_ctx, case, prec):
    from paper_1208_4093_gb300 import capi
    nx, ny, sx, sy, ov = case
    if prec == 0 and min(nx, sx + 2 * ov) > 64:
        pytest.skip("FP64 regions are at most 64 nodes wide")
    ea = ea_lognormal(nx, ny, 11)
    tr = truss.Truss(nx, ny, ea)
    g = hms.SetGrid(nx, ny, sx, sy)
    rng = np.random.default_rng(nx * 1000 + ny)
    r = tr.residual(tr.free * loads(nx, ny, 7).reshape(-1), tr.free * rng.standard_normal(tr.ndof))
    want = hms.LocalFactors(tr, g, overlap=ov).relax(r)
    outs = []
    for kw in (dict(), dict(relax_threads=64, relax_copies=1), dict(relax_threads=256, relax_copies=1)):
        pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, ea=ea, precision=prec, relax_overlap=ov, **kw)
        try:
            d, P = np.empty(tr.ndof), np.empty(9 * g.M)
            capi.hms_relax(hms_ctx, pr, r, d, P)
            outs.append((d, P))
        finally:
            capi.hms_problem_destroy(pr)
    d, P = outs[0]
    assert rel(d, want) < (2e-5 if prec else 1e-11)
    assert rel(P, hms.modes(tr, g, d).T @ r) < 1e-12
    for d2, P2 in outs[1:]:
        assert np.array_equal(d, d2) and np.array_equal(P, P2)


@pytest.mark.parametrize("nx,ny,sx,sy", [(31, 29, 11, 9), (50, 42, 24, 20)])
def test_force_relax_step(hms_ctx, nx, ny, sx, sy):
    from paper_1208_4093_gb300 import capi
    ea = ea_lognormal(nx, ny, 13)
    tr = truss.Truss(nx, ny, ea)
    g = hms.SetGrid(nx, ny, sx, sy)
    r = tr.free * np.random.default_rng(5).standard_normal(tr.ndof)
    pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, ea=ea, mode_mask=0xFFF)
    try:
        d = np.empty(tr.ndof)
        capi.hms_relax_force(hms_ctx, pr, r, d)
    finally:
        capi.hms_problem_destroy(pr)
    assert rel(d, hms.ForceFactors(tr, g).relax(r)) < 1e-8  # as in test_gpu_force


@pytest.mark.parametrize("nx,ny,sx,sy", [(64, 64, 16, 16), (71, 45, 16, 12), (140, 20, 64, 7)])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_class_relax_forms(hms_ctx, nx, ny, sx, sy, prec):
    """Class factors: sets sharing a dissected factor equal sets with their own
    bit for bit (the same k^Inner); the batched form (relax_balance = 1) to
    rounding."""
    from paper_1208_4093_gb300 import capi
    tr = truss.Truss(nx, ny)
    g = hms.SetGrid(nx, ny, sx, sy)
    r = tr.free * np.random.default_rng(9).standard_normal(tr.ndof)
    outs = []
    for kw in (dict(), dict(class_factors=1), dict(class_factors=1, relax_balance=1)):
        pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, precision=prec, relax_threads=256, relax_copies=1, **kw)
        try:
            d, P = np.empty(tr.ndof), np.empty(9 * g.M)
            capi.hms_relax(hms_ctx, pr, r, d, P)
            outs.append((d, P))
        finally:
            capi.hms_problem_destroy(pr)
    assert np.array_equal(outs[0][0], outs[1][0]) and np.array_equal(outs[0][1], outs[1][1])
    assert rel(outs[2][0], hms.LocalFactors(tr, g).relax(r)) < (2e-5 if prec else 1e-11)
