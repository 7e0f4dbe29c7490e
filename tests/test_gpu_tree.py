"""The tree of swept fronts of Eq. 8 (coarse_tree.cu; automatic choice and
coarse_factor = 6) at the sizes where its layout changes: one front (up to 256
unknowns) and more, fronts of one to eighteen 32-unknown block rows, boxes cut
once or twice, one CTA or a cluster per front, nine and twelve modes.

Each refined solution must meet the Galerkin condition (Eq. 5) to the oracle's
accuracy, as in test_gpu_nd, and whole solves the direct solve; batches in
lockstep must equal solo solves bit for bit.
"""
import numpy as np
import pytest

from oracle import direct, hms, truss
from workloads import batched_lattices, ea_lognormal, loads

pytestmark = pytest.mark.gpu


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


# set grids: 1x1, one row, one column, 256 unknowns and just above (28 sets: 252;
# 29: 261), leaves of four sets and one more, ragged, elongated
GRIDS = [(1, 1), (7, 1), (1, 30), (7, 4), (29, 1), (5, 6), (4, 8), (9, 5), (13, 11), (40, 3)]


@pytest.mark.parametrize("mx,my", GRIDS)
@pytest.mark.parametrize("q", [9, 12])
def test_tree_coarse_solve(hms_ctx, mx, my, q):
    from paper_1208_4093_gb300 import capi
    sx, sy = 5, 4
    nx, ny = mx * sx - (mx > 1), my * sy - (my > 1)
    ea = ea_lognormal(nx, ny, 31)
    tr = truss.Truss(nx, ny, ea)
    g = hms.SetGrid(nx, ny, sx, sy)
    pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, ea=ea, coarse_factor=6, coarse_solves=6,
                                 mode_mask=0xFFF if q == 12 else 0x1FF)
    try:
        rng = np.random.default_rng(mx * 100 + my)
        n = q * g.M
        # a system of the set grid's block pattern, unit diagonal times scales
        # over six decades, one mode of the first set vanishing
        A = np.zeros((n, n))
        for I in range(g.M):
            for J in range(I + 1):
                if abs(I % mx - J % mx) <= 1 and abs(I // mx - J // mx) <= 1:
                    A[I * q:(I + 1) * q, J * q:(J + 1) * q] = 0.02 * rng.standard_normal((q, q))
        A = np.tril(A, -1)
        A = A + A.T + np.eye(n)
        s = 10.0 ** rng.uniform(-3, 3, n)
        unit = A
        A = s[:, None] * A * s[None, :]
        A[2, :] = A[:, 2] = 0.0
        b = s * rng.standard_normal(n)
        b[2] = 0.0
        a = np.empty(n)
        dr = np.zeros(n, np.int32)
        capi.hms_coarse_solve(hms_ctx, pr, A, b, a, dr)
        keep = np.arange(n) != 2
        assert np.array_equal(dr != 0, ~keep) and a[2] == 0.0
        # unit-diagonal system, condition number below 10: refinement ends at
        # 1e-14 max |b|, 1e-12 leaves room for the norm (the reference solves the
        # unit-diagonal system too: the scaled one costs LU three digits)
        assert rel(s[keep] * a[keep], np.linalg.solve(unit[np.ix_(keep, keep)], (b / s)[keep])) < 1e-12
    finally:
        capi.hms_problem_destroy(pr)


@pytest.mark.parametrize("nx,ny,sx,sy", [(280, 232, 8, 8), (160, 400, 8, 8), (97, 61, 6, 6)],
                         ids=["35x29_sets", "20x50_sets", "17x11_sets"])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_tree_whole_solve(hms_ctx, nx, ny, sx, sy, prec):
    from paper_1208_4093_gb300 import capi
    ea = ea_lognormal(nx, ny, 37)
    tr = truss.Truss(nx, ny, ea)
    p = tr.free * loads(nx, ny, 12).reshape(-1)
    pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, ea=ea, precision=prec, tol=1e-11, max_iter=3000)
    try:
        out = np.empty((1, tr.ndof))
        capi.hms_solve(hms_ctx, pr, p.reshape(1, -1), out)
        assert rel(out[0], direct.sparse_solve(tr, p)) < (1e-8 if prec else 1e-9)
        assert capi.hms_problem_device_bytes(pr) <= capi.hms_problem_estimate_bytes(
            hms_ctx, nx, ny, sx, sy, ea=ea, precision=prec, tol=1e-11, max_iter=3000)
    finally:
        capi.hms_problem_destroy(pr)


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_tree_lockstep_equals_streams_and_solo(hms_ctx, prec):
    """Trees of different depth and cluster sizes, and a band factor beside
    them, in one lockstep batch."""
    from paper_1208_4093_gb300 import capi
    lats = batched_lattices(count=8, seed=17, side_min=24, side_max=160, nrhs_max=2)
    prs = [capi.hms_problem_create(hms_ctx, l.nx, l.ny, 12, 12, precision=prec, tol=1e-9, max_iter=4000,
                                   coarse_factor=4 if k == 3 else 0) for k, l in enumerate(lats)]
    try:
        ps = [l.load_array() for l in lats]
        res = {}
        for mode in (capi.HMS_BATCH_LOCKSTEP, capi.HMS_BATCH_STREAMS):
            capi.hms_context_set_batch_mode(hms_ctx, mode)
            res[mode] = [np.empty_like(p) for p in ps]
            capi.hms_solve_batch(hms_ctx, prs, ps, res[mode])
        for l, pr, p, a, b in zip(lats, prs, ps, *res.values()):
            solo = np.empty_like(p)
            capi.hms_solve(hms_ctx, pr, p, solo)
            assert np.array_equal(a, solo) and np.array_equal(b, solo), (l.nx, l.ny)
    finally:
        capi.hms_context_set_batch_mode(hms_ctx, capi.HMS_BATCH_AUTO)
        for pr in prs:
            capi.hms_problem_destroy(pr)
