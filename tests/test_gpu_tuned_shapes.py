"""Which problems of a context share a relaxation launch shape picked by timing: those
for which the choice is the same one.  More sets than SMs let the FP64 relaxation's
smaller ring put two sets on an SM, twelve modes relax every set twice in a launch, and
a last column of sets too narrow for two copies per matrix leaves fewer candidates (and
makes a choice of two copies impossible to launch for the row substitution)."""
import numpy as np
import pytest

from oracle import direct, truss
from workloads import loads

pytestmark = pytest.mark.gpu


def shapes_after(ctx, *args, **kw):
    from paper_1208_4093_gb300 import capi
    pr = capi.hms_problem_create(ctx, *args, **kw)
    try:
        assert capi.hms_problem_relax_threads(pr) in (64, 128, 256)
        if args[:2] == (66, 40):  # the ragged lattice is also solved with the choice it got
            p = loads(66, 40, 5).reshape(1, -1)
            u = np.empty_like(p)
            capi.hms_solve(ctx, pr, p, u)
            tr = truss.Truss(66, 40)
            ref = direct.cholesky_solve(tr, tr.free * p[0])
            assert np.linalg.norm(u[0] - ref) < 1e-8 * np.linalg.norm(ref)
    finally:
        capi.hms_problem_destroy(pr)
    return capi.hms_context_tuned_shapes(ctx)


def test_the_choice_is_kept_for_the_load_it_was_timed_at():
    from paper_1208_4093_gb300 import capi
    ctx = capi.hms_context_create(0)
    try:
        import torch
        nsm = torch.cuda.get_device_properties(0).multi_processor_count
        tile = (16, 12)

        def lattice(sets):  # one row of sets
            return sets * tile[0], tile[1], *tile
        assert capi.hms_context_tuned_shapes(ctx) == 0
        assert shapes_after(ctx, *lattice(4)) == 1
        assert shapes_after(ctx, *lattice(nsm)) == 1          # one set per SM, as before
        assert shapes_after(ctx, *lattice(nsm + 1)) == 2      # two on some
        assert shapes_after(ctx, *lattice(2 * nsm)) == 2
        assert shapes_after(ctx, *lattice(nsm), mode_mask=0xFFF) == 2  # two relaxations per set
        assert shapes_after(ctx, *lattice(4 * nsm)) == 3
        assert shapes_after(ctx, *lattice(9 * nsm)) == 3      # four and more alike
        assert shapes_after(ctx, *lattice(4)) == 3
    finally:
        capi.hms_context_destroy(ctx)


@pytest.mark.parametrize("balance", [0, 1])
def test_a_narrow_last_column_is_timed_by_itself(balance):
    from paper_1208_4093_gb300 import capi
    ctx = capi.hms_context_create(0)
    try:
        kw = dict(relax_balance=balance, tol=1e-10, max_iter=2000)
        assert shapes_after(ctx, 64, 40, 32, 20, **kw) == 1
        assert shapes_after(ctx, 66, 40, 32, 20, **kw) == 2  # last sets two nodes wide: one copy only
    finally:
        capi.hms_context_destroy(ctx)
