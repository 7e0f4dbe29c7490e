"""The dissected factors of small set tiles are larger than those of the row
substitution (padding to 32 lanes).  Where only the smaller ones fit -- a server's
budget, the device's free memory -- the problem runs the row substitution instead of
being refused."""
import numpy as np
import pytest

from workloads import ea_lognormal, loads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [1, 3])
def test_a_request_that_fits_the_budget_only_by_rows_is_served(hms_ctx, nrhs):
    from paper_1208_4093_gb300 import capi
    nx, ny, sx, sy = 90, 80, 9, 8  # 100 sets of 72 nodes
    kw = dict(ea=ea_lognormal(nx, ny, 3), tol=1e-9, max_iter=3000)
    p = np.concatenate([loads(nx, ny, k).reshape(1, -1) for k in range(nrhs)])
    rows = capi.hms_problem_estimate_bytes(hms_ctx, nx, ny, sx, sy, relax_balance=1, **kw)
    tree = capi.hms_problem_estimate_bytes(hms_ctx, nx, ny, sx, sy, **kw)
    assert tree > rows
    # a clone's own bytes, by creating one
    pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, relax_balance=1, **kw)
    cl = capi.hms_problem_clone(hms_ctx, pr)
    clone = capi.hms_problem_device_bytes(cl)
    capi.hms_problem_destroy(cl)
    capi.hms_problem_destroy(pr)
    rows += (nrhs - 1) * clone
    tree += (nrhs - 1) * clone
    got = {}
    for budget, form in ((rows, 1), ((rows + tree) // 2, 1), (tree, 0)):
        want = np.empty_like(p)
        pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, relax_balance=form, **kw)
        try:
            assert capi.hms_problem_relax_form(pr) == form
            capi.hms_solve(hms_ctx, pr, p, want)
        finally:
            capi.hms_problem_destroy(pr)
        srv = capi.hms_server_create(hms_ctx, budget, max_active=4)
        try:
            rid = capi.hms_server_submit(hms_ctx, srv, nx, ny, sx, sy, p, **kw)
            done = []
            for _ in range(5000):
                d, active, queued, used = capi.hms_server_step(hms_ctx, srv)
                done += d
                assert used <= budget
                if active == 0 and queued == 0:
                    break
            assert done == [rid]
            u = np.empty_like(p)
            capi.hms_server_take(hms_ctx, srv, rid, u)
            assert np.array_equal(u, want)
            got[budget] = u
        finally:
            capi.hms_server_destroy(srv)
    assert not np.array_equal(got[rows], got[tree])  # the forms differ in rounding
    srv = capi.hms_server_create(hms_ctx, rows - 1, max_active=4)
    try:
        with pytest.raises(capi.HmsError) as e:
            capi.hms_server_submit(hms_ctx, srv, nx, ny, sx, sy, p, **kw)
        assert e.value.status == capi.HMS_ERR_OOM
    finally:
        capi.hms_server_destroy(srv)


def test_a_problem_that_fits_the_free_memory_only_by_rows_is_created(hms_ctx):
    import torch
    from paper_1208_4093_gb300 import capi
    nx, ny, sx, sy = 1000, 780, 10, 13  # 6000 sets of 130 nodes
    kw = dict(tol=0.0, max_iter=2)
    p = loads(nx, ny, 1).reshape(1, -1)
    rows = capi.hms_problem_estimate_bytes(hms_ctx, nx, ny, sx, sy, relax_balance=1, **kw)
    tree = capi.hms_problem_estimate_bytes(hms_ctx, nx, ny, sx, sy, **kw)
    assert tree - rows > 400 << 20
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(free - (rows + tree) // 2, dtype=torch.uint8, device="cuda")
    try:
        assert rows <= capi.hms_problem_estimate_bytes(hms_ctx, nx, ny, sx, sy, **kw) < tree
        pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, **kw)
        try:
            assert capi.hms_problem_relax_form(pr) in (capi.HMS_RELAX_ROWS, capi.HMS_RELAX_BALANCED)
            low = np.empty_like(p)
            capi.hms_solve(hms_ctx, pr, p, low, allow_no_convergence=True)
        finally:
            capi.hms_problem_destroy(pr)
    finally:
        del hold
        torch.cuda.empty_cache()
    pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy, **kw)
    try:
        assert capi.hms_problem_relax_form(pr) == capi.HMS_RELAX_DISSECTED
        u = np.empty_like(p)
        capi.hms_solve(hms_ctx, pr, p, u, allow_no_convergence=True)
    finally:
        capi.hms_problem_destroy(pr)
    # two updates from rounding: FP64 local solves agree to 1e-11 (test_gpu_parity)
    assert np.linalg.norm(u - low) < 1e-9 * np.linalg.norm(u)


def test_work_space_of_the_factorisation_counts(hms_ctx):
    """24 x 20-node tiles: the factors are smaller than the row substitution's, but with
    the work space that their factorisation keeps the problem is larger."""
    import torch
    from paper_1208_4093_gb300 import capi
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    nx, ny, sx, sy = 24 * nsm, 20, 24, 20
    rows = capi.hms_problem_estimate_bytes(hms_ctx, nx, ny, sx, sy, relax_balance=1)
    tree = capi.hms_problem_estimate_bytes(hms_ctx, nx, ny, sx, sy)
    assert tree > rows
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - tree - (128 << 20), dtype=torch.uint8, device="cuda")
    try:
        assert capi.hms_problem_estimate_bytes(hms_ctx, nx, ny, sx, sy) == rows
        pr = capi.hms_problem_create(hms_ctx, nx, ny, sx, sy)
        try:
            assert capi.hms_problem_relax_form(pr) == capi.HMS_RELAX_ROWS
        finally:
            capi.hms_problem_destroy(pr)
    finally:
        del hold
        torch.cuda.empty_cache()
