"""The blocked float64 inverse on blocks whose every pivot is off the diagonal.

A strictly dominant system with the point rows of every block row permuted (A_i, B_i, C_i and b_i alike):
the solution and the condition number stay those of the dominant system, but every pivot of every block
inverse is an exchange.  Tolerance: the float64 path's 1e-12 of the oracle, the dominant systems being well
conditioned (1.1 to 1.3)."""
import numpy as np
import pytest

from oracle import dm_oracle as o
from paper_1505_06864_gb300 import workloads as w

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module")
def dm():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1505_06864_gb300 import build
    build.build()
    from paper_1505_06864_gb300 import dm as D
    return D


def permuted_system(N, m, r, seed):
    s = w.dominant_system(N, m, r, seed)
    rng = np.random.default_rng(seed)
    for i in range(N):
        p = rng.permutation(m)
        for X in (s.A, s.B, s.C, s.b):
            X[i] = X[i][p]
    return s


# block sizes around the subpanels (8), the panels (32), the chain's warps (32 rows each) and its register
# rows (one to 256, two above)
@pytest.mark.parametrize("N,m,r,P,levels", [(9, 8, 1, 2, 1), (9, 24, 2, 3, 1), (9, 40, 1, 2, 1), (12, 64, 3, 3, 1),
                                            (9, 128, 1, 3, 1), (7, 136, 2, 2, 1), (7, 248, 1, 2, 1),
                                            (7, 256, 1, 3, 1),
                                            # no multiples of 8 (padded slice rows, narrow last panels), above 256
                                            (9, 9, 1, 2, 1), (12, 31, 3, 3, 1), (9, 33, 1, 2, 1), (9, 100, 2, 3, 1),
                                            (9, 129, 1, 2, 1), (7, 201, 2, 3, 1), (7, 257, 1, 2, 1),
                                            (7, 400, 2, 3, 1), (5, 511, 1, 2, 1), (5, 512, 1, 2, 1)])
def test_every_pivot_exchanged(dm, N, m, r, P, levels):
    s = permuted_system(N, m, r, m + N)
    plan = dm.dm_plan(N, m, r, P, levels, "fp64")
    try:
        dm.dm_factor(plan, s.A, s.B, s.C)
        x = np.zeros_like(s.b)
        dm.dm_solve(plan, s.b, x)
    finally:
        dm.dm_destroy(plan)
    xref = o.dm(s.A, s.B, s.C, s.b, P)
    assert np.all(np.isfinite(x))
    assert np.all(np.max(np.abs(x - xref), axis=(0, 1)) <= TOL * np.max(np.abs(xref), axis=(0, 1)))
    assert o.rel_err(x, xref) <= TOL


def test_plan_without_room_for_slices_keeps_the_float64_pipe(dm):
    """A float64 plan with m % 8 != 0 whose digit slices do not fit is planned without them."""
    import torch
    N, m = 2500, 100
    entries = N * m * m
    plan = dm.dm_plan(N, m, 1, 16, 1, "fp64")
    sliced = dm.dm_plan_query(plan)["device_bytes"]
    dm.dm_destroy(plan)
    assert sliced > 70 * entries  # factors 32, slices 44 bytes per entry of a block
    free, _ = torch.cuda.mem_get_info()
    reserve = 1 << 30  # what dm_plan leaves free
    hold = torch.empty(free - reserve - 55 * entries, dtype=torch.uint8, device="cuda")
    try:
        plan = dm.dm_plan(N, m, 1, 16, 1, "fp64")
        assert dm.dm_plan_query(plan)["device_bytes"] < 40 * entries
        dm.dm_destroy(plan)
    finally:
        del hold
        torch.cuda.empty_cache()
