"""Float32 block inverse with every pivot exchanged: block sizes around its panels of 8 columns, its warps of 32 rows
and one or two rows per lane, up to the largest it takes (224) and the next.  Tolerance: the float32 factor is refined
with float64 residuals to the mixed path's 1e-10 of the oracle; the inverse of these well-conditioned blocks
(condition below 1e2) is within m 2^-24 of exact to a factor of 1e2, 2e-3 at most, so a correction is followed by one
at least 1 / 2e-3 times smaller and 1e-12 is reached in 12 / 2.7, at most 5, iterations."""
import numpy as np
import pytest

from oracle import dm_oracle as o
from test_gpu_blocked_inverse import dm, permuted_system  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 7, 8, 9, 31, 32, 33, 63, 65, 96, 97, 127, 128, 129, 160, 223, 224, 225])
def test_every_pivot_exchanged(dm, m):  # noqa: F811
    s = permuted_system(9, m, 2, 7 * m)
    plan = dm.dm_plan(9, m, 2, 3, 1, "fp32")
    try:
        dm.dm_factor(plan, s.A, s.B, s.C)
        x = np.zeros_like(s.b)
        dm.dm_solve(plan, s.b, x)
        info = dm.dm_plan_query(plan)
    finally:
        dm.dm_destroy(plan)
    assert np.all(np.isfinite(x))
    assert o.rel_err(x, o.dm(s.A, s.B, s.C, s.b, 3)) <= 1e-10
    assert info["last_iters"] <= 5 and info["last_correction"] <= 1e-12
