"""The solves by the tree of fronts on every cluster size that a device may be able to
place: the plan takes the largest one allowed, and the iterates are the same bits.
Without any the problem takes the form it would take if the fronts did not fit."""
import numpy as np
import pytest

from workloads import ea_lognormal, loads

pytestmark = pytest.mark.gpu

# set grid 1 x 1 (nine unknowns: one CTA), 3 x 4 (108: four) and 17 x 11 (1683: sixteen)
CASES = [(16, 12, 16, 12, 1), (18, 24, 6, 6, 4), (97, 61, 6, 6, 16)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[:4])))
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("mask", [0x1FF, 0xFFF], ids=["q9", "q12"])
def test_every_cluster_size_gives_the_same_bits(hms_ctx, case, prec, mask):
    from paper_1208_4093_gb300 import capi
    nx, ny, sx, sy, most = case
    if mask == 0xFFF and (nx - 1) % sx == 0:
        sx, sy = 7, 7  # one-node-wide last sets cannot be cut free
    if mask == 0xFFF and most == 4:
        most = 8  # 144 unknowns
    ea = ea_lognormal(nx, ny, 5)
    p = loads(nx, ny, 2).reshape(1, -1)
    outs = []
    try:
        for limit in (16, 8, 4, 2, 1):
            capi.hms_context_set_tree_cluster(hms_ctx, limit)
            pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, ea=ea, precision=prec, mode_mask=mask,
                                         coarse_factor=6, tol=0.0, max_iter=4)
            try:
                assert capi.hms_problem_coarse_form(pr) == (capi.HMS_COARSE_TREE, min(limit, most))
                u = np.empty_like(p)
                capi.hms_solve(hms_ctx, pr, p, u, allow_no_convergence=True)
                outs.append(u)
            finally:
                capi.hms_problem_destroy(pr)
    finally:
        capi.hms_context_set_tree_cluster(hms_ctx, 16)
    assert np.all(np.isfinite(outs[0])) and np.any(outs[0] != 0.0)
    for u in outs[1:]:
        assert np.array_equal(u, outs[0])


@pytest.mark.parametrize("factor", [0, 6])
def test_without_a_cluster_no_tree(hms_ctx, factor):
    from paper_1208_4093_gb300 import capi
    nx, ny, sx, sy = 60, 46, 6, 6
    args = dict(coarse_factor=factor, tol=1e-11, max_iter=2000)
    p = loads(nx, ny, 2).reshape(1, -1)
    outs = []
    try:
        for limit in (16, 0):
            capi.hms_context_set_tree_cluster(hms_ctx, limit)
            pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, **args)
            try:
                form, ctas = capi.hms_problem_coarse_form(pr)
                if limit:
                    assert form == capi.HMS_COARSE_TREE and ctas > 0
                else:
                    assert ctas == 0
                    assert form == capi.HMS_COARSE_PANELS if factor == 6 else form <= capi.HMS_COARSE_BAND_TWO_SIDED
                assert capi.hms_problem_device_bytes(pr) <= capi.hms_problem_estimate_bytes(hms_ctx, nx, ny, sx, sy,
                                                                                             **args)
                u = np.empty_like(p)
                capi.hms_solve(hms_ctx, pr, p, u)
                outs.append(u)
            finally:
                capi.hms_problem_destroy(pr)
    finally:
        capi.hms_context_set_tree_cluster(hms_ctx, 16)
    # both converged to R1 < 1e-11; the bar of test_gpu_parity for converged displacements
    assert np.linalg.norm(outs[1] - outs[0]) < 1e-9 * np.linalg.norm(outs[0])


def test_bad_limits_are_refused(hms_ctx):
    from paper_1208_4093_gb300 import capi
    for bad in (-1, 3, 12, 17, 32):
        with pytest.raises(capi.HmsError) as e:
            capi.hms_context_set_tree_cluster(hms_ctx, bad)
        assert e.value.status == capi.HMS_ERR_ARG
