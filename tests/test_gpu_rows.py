"""The row substitution (relax.cu; relax_balance = 1) and the batched class factors
(relax_class.cu) on set tiles of more than 64 nodes, where nested dissection is the
usual choice: the checks of the other files -- steps against the oracle, the same bits
for every CTA size and copies per matrix, grown regions, cut-free sets, the bounded
wait -- with relax_balance = 1 and every problem's form asserted.  Tiles whose
dissected factors would not fit still run these."""
import pytest

import test_gpu_autotune
import test_gpu_boundary
import test_gpu_class
import test_gpu_force
import test_gpu_overlap
import test_gpu_rtree

pytestmark = pytest.mark.gpu


@pytest.fixture
def rows_ctx(hms_ctx, monkeypatch):
    """The context; problems are created with relax_balance = 1 and must run it."""
    from paper_1208_4093_gb300 import capi
    create = capi.hms_problem_create

    def checked(*args, **kw):
        pr = create(*args, **dict(kw, relax_balance=1))
        want = capi.HMS_RELAX_CLASS_BATCHES if kw.get("class_factors") else capi.HMS_RELAX_ROWS
        if capi.hms_problem_relax_form(pr) != want:
            capi.hms_problem_destroy(pr)
            raise AssertionError("not the row substitution")
        return pr
    monkeypatch.setattr(capi, "hms_problem_create", checked)
    return hms_ctx


def test_the_forms_are_told_apart(hms_ctx):
    from paper_1208_4093_gb300 import capi
    for args, kw, want in (((64, 64, 16, 16), {}, capi.HMS_RELAX_DISSECTED),
                           ((64, 64, 16, 16), dict(class_factors=1), capi.HMS_RELAX_DISSECTED),
                           ((64, 64, 16, 16), dict(relax_balance=1), capi.HMS_RELAX_ROWS),
                           ((32, 32, 8, 8), {}, capi.HMS_RELAX_ROWS),
                           ((128, 128, 8, 8), dict(relax_balance=2), capi.HMS_RELAX_BALANCED),
                           ((32, 32, 8, 8), dict(class_factors=1), capi.HMS_RELAX_CLASS_BATCHES)):
        pr = capi.hms_problem_create(hms_ctx, *args, **kw)
        try:
            assert capi.hms_problem_relax_form(pr) == want
        finally:
            capi.hms_problem_destroy(pr)


@pytest.mark.parametrize("shape", test_gpu_autotune.SHAPES, ids=lambda s: f"{s[0]}x{s[1]}_sets{s[2]}x{s[3]}")
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_every_cta_size_gives_the_same_bits(rows_ctx, shape, prec):
    test_gpu_autotune.test_every_cta_size_gives_the_same_bits(rows_ctx, shape, prec)


@pytest.mark.parametrize("case", test_gpu_rtree.CASES, ids=["x".join(map(str, c)) for c in test_gpu_rtree.CASES])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_relax_step(rows_ctx, case, prec):
    test_gpu_rtree.test_relax_step(rows_ctx, case, prec)


@pytest.mark.parametrize("case", test_gpu_overlap.CASES, ids=lambda c: c[0])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_grown_regions(rows_ctx, case, prec):
    test_gpu_overlap.test_overlap_relax_step(rows_ctx, case, prec)
    test_gpu_overlap.test_overlap_full_solve(rows_ctx, case, prec)


def test_grown_regions_launch_shapes_batches_and_copies(rows_ctx):
    test_gpu_overlap.test_overlap_launch_shapes_and_batch_agree(rows_ctx)
    test_gpu_overlap.test_overlap_after_the_same_set_shape_without(rows_ctx)


@pytest.mark.parametrize("nx,ny,sx,sy", [(31, 29, 11, 9), (50, 42, 24, 20)])
def test_cut_free_sets(rows_ctx, nx, ny, sx, sy):
    test_gpu_rtree.test_force_relax_step(rows_ctx, nx, ny, sx, sy)


@pytest.mark.parametrize("prec", [0, 1])
def test_twelve_modes_reach_the_direct_solution(rows_ctx, prec):
    case = ("tiles11x9", 31, 29, 11, 9, True, None)
    test_gpu_force.test_q12_solve_reaches_direct_solution(rows_ctx, case, prec)


@pytest.mark.parametrize("precision", [0, 1])
def test_the_bounded_wait_drains(rows_ctx, precision):
    test_gpu_boundary.test_relaxation_timeout_is_reported_and_recovers(rows_ctx, precision)


@pytest.mark.parametrize("case", test_gpu_class.CASES, ids=[c[0] for c in test_gpu_class.CASES])
@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_class_batches(rows_ctx, case, prec):
    test_gpu_class.test_class_relax_step(rows_ctx, case, prec)
