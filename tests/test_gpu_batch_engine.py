"""Which engine a batch runs on: lockstep and streams give the same bits, so the choice
is one of time.  With trees of fronts in the batch lockstep is the faster one for
lattices of about one size and for more problems than two per stream; unlike lattices
go on at their own pace on streams."""
import numpy as np
import pytest

from workloads import loads

pytestmark = pytest.mark.gpu


@pytest.fixture
def batch(hms_ctx):
    from paper_1208_4093_gb300 import capi
    prs = []

    def make(shapes, **kw):
        new = [capi.hms_problem_create(hms_ctx, nx, ny, 12, 12, tol=1e-9, max_iter=4000, **kw) for nx, ny in shapes]
        prs.extend(new)
        return new
    yield make
    capi.hms_context_set_batch_mode(hms_ctx, capi.HMS_BATCH_AUTO)
    for pr in prs:
        capi.hms_problem_destroy(pr)


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "mixed"])
def test_engine_by_sizes(hms_ctx, batch, prec):
    from paper_1208_4093_gb300 import capi
    big, small = (96, 96), (24, 24)
    alike = batch([big, (96, 48), big], precision=prec)           # twice the nodes
    unlike = batch([big, (96, 47), small], precision=prec)
    band = batch([big, small], precision=prec, coarse_factor=4)   # as ever
    many = [capi.hms_problem_clone(hms_ctx, unlike[2]) for _ in range(128)]
    LOCK, STREAMS = capi.HMS_BATCH_LOCKSTEP, capi.HMS_BATCH_STREAMS
    try:
        for prs, auto in ((alike, LOCK), (unlike, STREAMS), (unlike[:2], STREAMS), (unlike[:1], LOCK), (band, LOCK),
                          (band + unlike[2:], STREAMS), (unlike[:1] + many[:127], STREAMS), (unlike[:1] + many, LOCK),
                          (many, LOCK)):
            capi.hms_context_set_batch_mode(hms_ctx, capi.HMS_BATCH_AUTO)
            assert capi.hms_batch_engine(hms_ctx, prs) == auto, (len(prs), auto)
            for mode in (LOCK, STREAMS):  # a mode that is set stands
                capi.hms_context_set_batch_mode(hms_ctx, mode)
                assert capi.hms_batch_engine(hms_ctx, prs) == mode
        # the automatic choice solves as either engine does
        ps = [loads(nx, ny, 3).reshape(1, -1) for nx, ny in (big, (96, 47), small)]
        res = []
        for mode in (capi.HMS_BATCH_AUTO, LOCK, STREAMS):
            capi.hms_context_set_batch_mode(hms_ctx, mode)
            res.append([np.empty_like(p) for p in ps])
            capi.hms_solve_batch(hms_ctx, unlike, ps, res[-1])
        for other in res[1:]:
            assert all(np.array_equal(a, b) for a, b in zip(res[0], other))
    finally:
        for pr in many:
            capi.hms_problem_destroy(pr)


def test_refusal_names_what_lockstep_needs(hms_ctx, batch):
    """Each refused batch breaks one condition of the message; a batch of trees breaks none."""
    from paper_1208_4093_gb300 import capi
    shape = (48, 144)
    tree, p = batch([shape])[0], loads(*shape, 3).reshape(1, -1)
    capi.hms_context_set_batch_mode(hms_ctx, capi.HMS_BATCH_LOCKSTEP)
    capi.hms_solve_batch(hms_ctx, [tree], [p], [np.empty_like(p)])
    for kw, need in ((dict(precision=1), "one precision"), (dict(coarse_solves=3), "one coarse_solves"),
                     (dict(mode_mask=0xFFF), "nine modes"), (dict(class_factors=1), "per-set factors"),
                     (dict(coarse_factor=5), "the tree of fronts or the one-SM FP32 factor")):
        other = batch([shape], **kw)[0]
        with pytest.raises(capi.HmsError) as e:
            capi.hms_solve_batch(hms_ctx, [tree, other], [p, p], [np.empty_like(p), np.empty_like(p)])
        assert e.value.status == capi.HMS_ERR_ARG
        assert need in capi.hms_last_error(hms_ctx), kw
