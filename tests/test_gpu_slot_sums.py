"""The sums over a set's threads that make up K_aa (Eq. 6) of a mixed problem with
twelve modes are FP64: only a thread's own products are FP32.

With EA = L = 1 and a delta^RF of even whole numbers along x every product of a bar
and its sum over a thread's nodes is a whole number below 2^24 (or an even one below
2^25), exact in FP32, so that entries without rounding are known: K[9][9] = sum s^2 and
K[9][2] = -sum s e_x^2 with s = e . (d_a - d_b) over the bars.  Adding up even two
threads' sums in FP32 rounds them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def bars(nx, ny):
    """(owner, other end, e_x) of every bar as index arrays, direction by direction."""
    j, i = np.mgrid[0:ny, 0:nx]
    off = j & 1
    for di, dj, ex in ((1, 0, 1.0), (off, 1, 0.5), (off - 1, 1, -0.5)):
        ib, jb = i + di, j + dj
        ok = (ib >= 0) & (ib < nx) & (jb < ny)
        yield (j * nx + i)[ok], (jb * nx + ib)[ok], ex


# One set of nx x ny nodes shared by 512 threads: n = 1 and 3 nodes of a thread at most.
# |d| <= t makes |s| <= 2 t along x and t for the other two bars of a node, so K[9][9]
# asks for 6 n t^2 < 2^24 and K[9][2] for 2 n t <= 2^25 (even) and n t <= 2^24.
@pytest.mark.parametrize("nx,ny,square,linear", [(22, 22, 1600, 1 << 23), (40, 37, 900, 5 << 20)])
def test_sums_over_threads_are_fp64(hms_ctx, nx, ny, square, linear):
    from paper_1208_4093_gb300 import capi
    pr = capi.hms_problem_create(hms_ctx, nx, ny, nx, ny, precision=1, mode_mask=0xFFF, bar_length=1.0)
    try:
        for top, row in ((square, 9), (linear, 2)):
            d = np.zeros((ny, nx, 2))
            # rows 0 (clamped) and 1 stay zero: no bar at a constrained DOF adds anything
            d[2:, :, 0] = 2 * np.random.default_rng(top).integers(-(top // 2), top // 2 + 1, (ny - 2, nx))
            K = np.empty((12, 12))
            capi.hms_coarse_matrix(hms_ctx, pr, np.concatenate([np.zeros(2 * nx * ny), d.reshape(-1)]), K)
            x = d[..., 0].reshape(-1)
            want = 0.0
            for a, b, ex in bars(nx, ny):
                s = ex * (x[a] - x[b])
                want += (s * s).sum() if row == 9 else -(s * ex * ex).sum()
            assert want != 0.0 and K[9, row] == want and K[row, 9] == want
    finally:
        capi.hms_problem_destroy(pr)
