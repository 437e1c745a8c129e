"""Blocks without a usable pivot (all zero, a zero column, NaN, infinite) in each block inverse, at one row and two rows
per lane: the factorisation names the block as singular or, where NaN lets pivots through, returns no finite
solution; the plan then takes a regular system as before.  (Every pivot search finds an eligible row, so the guard of
the row's number is not reached from here; these are the inputs closest to it.)"""
import numpy as np
import pytest

from oracle import dm_oracle as o
from paper_1505_06864_gb300 import workloads as w
from test_gpu_blocked_inverse import dm  # noqa: F401

pytestmark = pytest.mark.gpu


def spoil(s, i, kind):
    B = s.B.copy()
    if kind == "zero":
        B[i] = 0.0
        s.A[i] = 0.0
    elif kind == "column":
        B[i, :, s.m // 2] = 0.0
        s.A[i] = 0.0
    else:
        B[i] = np.nan if kind == "nan" else np.inf
    return B


@pytest.mark.parametrize("kind", ["zero", "column", "nan", "inf"])
@pytest.mark.parametrize("prec,m", [("fp64", 5), ("fp64", 32), ("fp64", 40), ("fp64", 129), ("fp64", 257),
                                    ("fp32", 33), ("fp32", 100), ("fp32", 129), ("fp32", 224)])
def test_no_usable_pivot(dm, prec, m, kind):  # noqa: F811
    s = w.dominant_system(6, m, 1, m)
    s0 = w.dominant_system(6, m, 1, m)
    B = spoil(s, 3, kind)
    plan = dm.dm_plan(6, m, 1, 1, 1, prec)
    x = np.zeros_like(s.b)
    try:
        try:
            dm.dm_factor(plan, s.A, B, s.C)
            assert kind in ("nan", "inf")
            try:
                dm.dm_solve(plan, s.b, x)
            except dm.DMError as e:
                assert e.code == dm.DM_ENOTCONV
            assert not np.all(np.isfinite(x))
        except dm.DMError as e:
            assert e.code == dm.DM_ESINGULAR and "block row 3" in str(e)
        dm.dm_factor(plan, s0.A, s0.B, s0.C)
        dm.dm_solve(plan, s0.b, x)
    finally:
        dm.dm_destroy(plan)
    assert o.rel_err(x, o.thomas(s0.A, s0.B, s0.C, s0.b)) <= (1e-12 if prec == "fp64" else 1e-10)
