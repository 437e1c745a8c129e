"""Float64 plans on systems whose equations or unknowns are of different scale.  Rows of [A_i B_i C_i | b_i] and
columns of T are scaled by powers of two over up to twelve decades, so the scaled system's solution is exactly the one
of the system it came from, unknown by unknown in its scale.

Tolerance: the error, so measured, of a plan on the float64 pipe (DM_PLAN_FP64_FMA), twice over, or 1e-14.  A numpy
restatement of both (block Thomas, m = 33 to 129, spans of 8, 16 and 40 binary orders on rows, columns and both) has the
digit-sliced elimination, equilibrated, at 0.1 to 1.5 times float64's error or below 2e-15; digits with one scale per
row and column give 1e-9 to 1e-5 at 40."""
import numpy as np
import pytest

from oracle import dm_oracle as o
from paper_1505_06864_gb300 import workloads as w
from test_gpu_blocked_inverse import dm  # noqa: F401

pytestmark = pytest.mark.gpu


def scaled(s, seed, rows, cols):
    """The system with equations / unknowns scaled by 2^-U(0, rows), 2^-U(0, cols); the unknowns' scales."""
    rng = np.random.default_rng(seed)
    R = 2.0 ** -np.rint(rng.uniform(0, rows, (s.N, s.m)))
    Q = 2.0 ** -np.rint(rng.uniform(0, cols, (s.N, s.m)))
    A, B, C = s.A * R[:, :, None], s.B * R[:, :, None] * Q[:, None, :], s.C * R[:, :, None]
    A[1:] *= Q[:-1, None, :]
    C[:-1] *= Q[1:, None, :]
    return A, B, C, s.b * R[:, :, None], Q[:, :, None]


def solution(dm, plan, A, B, C, b):
    x = np.zeros_like(b)
    try:
        dm.dm_factor(plan, A, B, C)
        dm.dm_solve(plan, b, x)
    finally:
        dm.dm_destroy(plan)
    return x


@pytest.mark.parametrize("rows,cols", [(40, 0), (0, 40), (40, 40), (16, 0), (0, 16)])
@pytest.mark.parametrize("kind,m,P,levels", [("dominant", 33, 3, 1), ("dominant", 100, 9, 2), ("dominant", 128, 3, 1),
                                             ("dominant", 256, 3, 1), ("dominant", 257, 2, 1), ("dominant", 400, 3, 1),
                                             ("laplace", 65, 3, 1), ("laplace", 100, 5, 1), ("banded", 72, 4, 1)])
def test_scaled_equations_and_unknowns(dm, kind, m, P, levels, rows, cols):  # noqa: F811
    N = 28 if P > 3 else 9
    make = {"dominant": w.dominant_system, "laplace": w.laplace_fill_system, "banded": w.pde_banded_system}[kind]
    s = make(N, m, 2, m)
    A, B, C, b, q = scaled(s, m + rows, rows, cols)
    ref = o.refine_truth(s.A, s.B, s.C, s.b)
    err = []
    for flags in (0, dm.DM_PLAN_FP64_FMA):
        x = solution(dm, dm.dm_plan_ex(N, m, 2, P, levels, "fp64", flags), A, B, C, b)
        err.append(float(np.max(np.abs(x * q - ref)) / np.max(np.abs(ref))))
    assert err[0] <= max(2 * err[1], 1e-14), err


@pytest.mark.parametrize("m", [33, 100, 300])
@pytest.mark.parametrize("k", [-990, 1014])
def test_ends_of_the_exponent_range(dm, m, k):  # noqa: F811
    """Blocks scaled as a whole: the pivots' reciprocals near the smallest and largest normal numbers."""
    s = w.dominant_system(9, m, 1, m)
    f = 2.0 ** k
    x = solution(dm, dm.dm_plan(9, m, 1, 3, 1, "fp64"), s.A * f, s.B * f, s.C * f, s.b * 2.0 ** -8 * f)
    assert o.rel_err(x * 2.0 ** 8, o.dm(s.A, s.B, s.C, s.b, 3)) <= 1e-12


@pytest.mark.parametrize("which", ["A", "C"])
def test_blocks_outside_the_system_are_not_read(dm, which):  # noqa: F811
    """A_1 and C_N belong to no equation: NaN there changes nothing."""
    s = w.dominant_system(12, 40, 1, 9)
    A, C = s.A.copy(), s.C.copy()
    if which == "A":
        A[0] = np.nan
    else:
        C[-1] = np.nan
    x = solution(dm, dm.dm_plan(12, 40, 1, 3, 1, "fp64"), A, s.B, C, s.b)
    assert o.rel_err(x, o.dm(s.A, s.B, s.C, s.b, 3)) <= 1e-12
