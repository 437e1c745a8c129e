"""The tensor-core residual at the edges of its tiles: 16-row tiles, groups of block rows per CTA, 8 columns per
class, and blocks whose addresses allow no 16-byte loads.  Bound and reference as in test_gpu_residual."""
import numpy as np
import pytest

from paper_1505_06864_gb300 import workloads as w
from test_gpu_residual import bound, dm, exact_residual  # noqa: F401

pytestmark = pytest.mark.gpu


def residual(dm, s, x, shift):
    """r = b - T x of a plan that borrows device blocks `shift` elements past a 16-byte boundary."""
    import torch

    def place(a):
        t = torch.empty(a.size + shift, dtype=torch.float64, device="cuda")[shift:]
        t.copy_(torch.from_numpy(np.ascontiguousarray(a)).reshape(-1))
        return t

    A, B, C = place(s.A), place(s.B), place(s.C)
    torch.cuda.synchronize()
    plan = dm.dm_plan(s.N, s.m, s.nrhs, 1, 1, "fp32")
    try:
        dm.dm_set_borrow_inputs(plan)
        dm.dm_set_residual(plan, "sliced")
        dm.dm_factor(plan, A, B, C)
        r = np.zeros_like(s.b)
        dm.dm_residual(plan, x, s.b, r)
        assert dm.dm_plan_query(plan)["residual_tc_systems"] == 1
    finally:
        dm.dm_destroy(plan)
    return r


@pytest.mark.parametrize("N,m,r", [(1, 1, 1), (9, 15, 8), (8, 16, 9), (17, 16, 1), (5, 31, 16), (6, 33, 7),
                                   (4, 63, 2), (3, 65, 9), (2, 127, 8), (3, 128, 1)])
@pytest.mark.parametrize("shift", [0, 1])
def test_tile_edges_and_alignment(dm, N, m, r, shift):  # noqa: F811
    s = w.dominant_system(N, m, r, 7 * m + r)
    rng = np.random.default_rng(m + r)
    x = rng.standard_normal(s.b.shape) * np.exp(rng.uniform(-3, 3, size=(1, 1, r)))
    err = np.abs(residual(dm, s, x, shift).astype(np.longdouble) - exact_residual(s.A, s.B, s.C, x, s.b))
    assert np.all(err.astype(np.float64) <= bound(s.A, s.B, s.C, x))
