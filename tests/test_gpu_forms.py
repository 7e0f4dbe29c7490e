"""Where the forms of the default path end: the last square set grid whose fronts fit
the tree in shared memory, and the last regions that nested dissection of a set takes;
one step further the problem still runs, in the other form."""
import numpy as np
import pytest

from workloads import loads

pytestmark = pytest.mark.gpu


def runs(ctx, nx, ny, sx, sy, **kw):
    """The forms of a problem that ran two updates to finite iterates."""
    from paper_1208_4093_gb300 import capi
    pr = capi.hms_problem_create(ctx, nx, ny, sx, sy, tol=0.0, max_iter=2, **kw)
    try:
        u = np.empty((1, 2 * nx * ny))
        capi.hms_solve(ctx, pr, loads(nx, ny, 1).reshape(1, -1), u, allow_no_convergence=True)
        assert np.all(np.isfinite(u)) and np.any(u != 0.0)
        return capi.hms_problem_coarse_form(pr)[0], capi.hms_problem_relax_form(pr)
    finally:
        capi.hms_problem_destroy(pr)


@pytest.mark.parametrize("last,mask", [(39, 0x1FF), (29, 0xFFF)], ids=["q9", "q12"])
def test_last_square_set_grid_of_the_tree(hms_ctx, last, mask):
    from paper_1208_4093_gb300 import capi
    for m, form in ((last, capi.HMS_COARSE_TREE), (last + 1, capi.HMS_COARSE_PANELS)):
        assert runs(hms_ctx, 3 * m, 3 * m, 3, 3, mode_mask=mask, coarse_factor=6)[0] == form


@pytest.mark.parametrize("tile,overlap,dissected", [((63, 63), 1, True), ((64, 64), 0, True), ((64, 64), 1, False),
                                                    ((64, 46), 1, True), ((64, 64), 8, False)])
def test_last_regions_of_the_dissection(hms_ctx, tile, overlap, dissected):
    from paper_1208_4093_gb300 import capi
    sx, sy = tile  # the middle one of three by three sets is grown on all sides
    form = runs(hms_ctx, 3 * sx, 3 * sy, sx, sy, relax_overlap=overlap, precision=1)[1]
    assert (form == capi.HMS_RELAX_DISSECTED) == dissected
