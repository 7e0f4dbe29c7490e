"""The fronts that are factored panel by panel from device memory (coarse_nd.cu) on
small set grids, where the tree of fronts in shared memory is the usual choice: the
step and whole-solve checks of test_gpu_nd and the step check of test_gpu_tree, for
nine and twelve modes, with every problem's form asserted.  The form is the only one
on set grids wider than about 40 sets (30 with twelve modes)."""
import pytest

import test_gpu_nd
import test_gpu_tree

pytestmark = pytest.mark.gpu


@pytest.fixture
def panels_ctx(hms_ctx, monkeypatch):
    """The context taking no tree of fronts; problems created must run the panels."""
    from paper_1208_4093_gb300 import capi
    create = capi.hms_problem_create

    def checked(*args, **kw):
        pr = create(*args, **kw)
        if capi.hms_problem_coarse_form(pr) != (capi.HMS_COARSE_PANELS, 0):
            capi.hms_problem_destroy(pr)
            raise AssertionError("not the panel-by-panel fronts")
        return pr
    monkeypatch.setattr(capi, "hms_problem_create", checked)
    capi.hms_context_set_tree_cluster(hms_ctx, 0)
    yield hms_ctx
    capi.hms_context_set_tree_cluster(hms_ctx, 16)


@pytest.mark.parametrize("case", test_gpu_nd.CASES, ids=lambda c: c[0])
def test_coarse_solve_matches_oracle(panels_ctx, case):
    test_gpu_nd.test_nd_coarse_solve_matches_oracle(panels_ctx, case)


@pytest.mark.parametrize("case", test_gpu_nd.CASES[:4] + test_gpu_nd.CASES[6:], ids=lambda c: c[0])
@pytest.mark.parametrize("precision", [0, 1])
def test_full_solve_and_trajectory(panels_ctx, case, precision):
    test_gpu_nd.test_nd_full_solve_and_trajectory(panels_ctx, case, precision)


@pytest.mark.parametrize("mx,my", test_gpu_tree.GRIDS)
@pytest.mark.parametrize("q", [9, 12])
def test_coarse_solve_of_block_systems(panels_ctx, mx, my, q):
    test_gpu_tree.test_tree_coarse_solve(panels_ctx, mx, my, q)
