"""Blocks of at most 32 whose pivots have a finite reciprocal that is not a normal number, or are not normal themselves:
accepted like any other (dm_factor refuses zero and non-finite pivots).  Sizes at the warps' column shares; the
solution of the system scaled by a power of two is that of the system itself."""
import numpy as np
import pytest

from oracle import dm_oracle as o
from paper_1505_06864_gb300 import workloads as w
from test_gpu_blocked_inverse import dm  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 3, 8, 9, 16, 17, 32])
@pytest.mark.parametrize("top", [1023, 1022])
def test_largest_pivots(dm, m, top):  # noqa: F811
    """The largest entry in [2^(top - 1), 2^top): pivots at and above 2^1022, reciprocals below 2^-1022."""
    s = w.dominant_system(9, m, 1, m)
    f = 2.0 ** (top - int(np.frexp(np.abs(s.B).max())[1]))
    plan = dm.dm_plan(9, m, 1, 3, 1, "fp64")
    x = np.zeros_like(s.b)
    try:
        dm.dm_factor(plan, s.A * f, s.B * f, s.C * f)
        dm.dm_solve(plan, s.b * 2.0 ** -8 * f, x)
    finally:
        dm.dm_destroy(plan)
    # a reciprocal between 2^-1024 and 2^-1022 keeps 50 bits or more: 8 units of 2^-50 per product with it, m of them
    assert o.rel_err(x * 2.0 ** 8, o.dm(s.A, s.B, s.C, s.b, 3)) <= 8 * m * 2.0 ** -50 + 1e-12


def test_smallest_pivots(dm):  # noqa: F811
    """2^-1023: below the smallest normal number, its reciprocal 2^1023 is finite."""
    B = np.full((4, 1, 1), 2.0 ** -1023)
    zero = np.zeros_like(B)
    plan = dm.dm_plan(4, 1, 1, 1, 1, "fp64")
    x = np.zeros((4, 1, 1))
    try:
        dm.dm_factor(plan, zero, B, zero)
        dm.dm_solve(plan, B * 0.5, x)
    finally:
        dm.dm_destroy(plan)
    assert np.array_equal(x, np.full_like(x, 0.5))
