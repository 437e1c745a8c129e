"""Float64 plans on systems whose equations or unknowns are of different scale.  Rows of [A_i B_i C_i | b_i] and
columns of T are scaled by powers of two over up to twelve decades, drawn per row or with a jump between the halves of
every block (two fields in different units), so the scaled system's solution is exactly the one of the system it came
from, unknown by unknown in its scale.

Tolerance: the error, so measured, of a plan on the float64 pipe (DM_PLAN_FP64_FMA), twice over, or 1e-14.  A numpy
restatement of both (block Thomas, m = 33 to 129, these scalings) has the digit-sliced elimination, equilibrated, at 0.1
to 1.5 times float64's error or below 1e-14 where it is kept; where the scales are ambiguous the level's products are
the float64 ones.  Digits with one scale per row and column give 1e-9 to 1e-4 at 40 binary orders."""
import numpy as np
import pytest

from oracle import dm_oracle as o
from paper_1505_06864_gb300 import workloads as w
from test_gpu_blocked_inverse import dm  # noqa: F401

pytestmark = pytest.mark.gpu


def exponents(rng, N, m, span, jump):
    if jump:
        return np.tile(np.where(np.arange(m) < m // 2, 0, -span), (N, 1))
    return -np.rint(rng.uniform(0, span, (N, m))).astype(int)


def scaled(s, seed, rows, cols, jump=False):
    """The system with equations / unknowns scaled over `rows` / `cols` binary orders; the unknowns' scales."""
    rng = np.random.default_rng(seed)
    R, Q = (np.ldexp(1.0, exponents(rng, s.N, s.m, span, jump)) for span in (rows, cols))
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


@pytest.mark.parametrize("rows,cols,jump", [(40, 0, False), (0, 40, False), (40, 40, False), (16, 0, False),
                                            (0, 16, False), (40, 0, True), (0, 40, True), (40, 40, True),
                                            (40, -40, True), (20, 0, True)])
@pytest.mark.parametrize("kind,m,P,levels", [("dominant", 33, 3, 1), ("dominant", 100, 9, 2), ("dominant", 128, 3, 1),
                                             ("dominant", 256, 3, 1), ("dominant", 257, 2, 1), ("dominant", 400, 3, 1),
                                             ("laplace", 65, 3, 1), ("laplace", 100, 5, 1), ("banded", 72, 4, 1),
                                             ("wide band", 100, 3, 1)])
def test_scaled_equations_and_unknowns(dm, kind, m, P, levels, rows, cols, jump):  # noqa: F811
    N = 28 if P > 3 else 9
    s = {"dominant": lambda: w.dominant_system(N, m, 2, m), "laplace": lambda: w.laplace_fill_system(N, m, 2, m),
         "banded": lambda: w.pde_banded_system(N, m, 2, m),
         "wide band": lambda: w.pde_banded_system(N, m, 2, m, hb=9)}[kind]()
    A, B, C, b, q = scaled(s, m + rows, rows, cols, jump)
    ref = o.refine_truth(s.A, s.B, s.C, s.b)
    err = []
    for flags in (0, dm.DM_PLAN_FP64_FMA):
        x = solution(dm, dm.dm_plan_ex(N, m, 2, P, levels, "fp64", flags), A, B, C, b)
        err.append(float(np.max(np.abs(x * q - ref)) / np.max(np.abs(ref))))
    assert err[0] <= max(2 * err[1], 1e-14), err


def panels(dm, plan, *blocks):
    """Launches of the digit-sliced inverse's panels in one factorisation."""
    dm.dm_profile(plan, True)
    dm.dm_factor(plan, *blocks)
    prof = dm.dm_profile(plan, False)
    return sum(v["launches"] for k, v in prof.items() if k.split("@")[0] == "inv_panel")


def test_result_does_not_depend_on_the_system_before(dm):  # noqa: F811
    """One plan through systems with digit and with float64 products in turn: the bits of a fresh plan each time
    (eager, captured and replayed launches), the products of an uneven system not tried in vain twice."""
    N, m = 40, 72
    s = w.pde_banded_system(N, m, 1, 3, hb=9)
    systems = [(s.A, s.B, s.C, s.b), scaled(s, 4, 40, 0, True)[:4], scaled(s, 5, 0, 30, True)[:4]]
    fresh = [solution(dm, dm.dm_plan(N, m, 1, 8, 2, "fp64"), *sy) for sy in systems]
    fma = solution(dm, dm.dm_plan_ex(N, m, 1, 8, 2, "fp64", dm.DM_PLAN_FP64_FMA), *systems[1])
    assert np.array_equal(fresh[1], fma)
    plan = dm.dm_plan(N, m, 1, 8, 2, "fp64")
    try:
        for k in (0, 1, 1, 2, 1, 0, 0, 2, 1, 0):
            x = np.zeros_like(s.b)
            dm.dm_factor(plan, *systems[k][:3])
            dm.dm_solve(plan, systems[k][3], x)
            assert np.array_equal(x, fresh[k]), k
        assert panels(dm, plan, *systems[0][:3]) > 0
        panels(dm, plan, *systems[1][:3])
        assert panels(dm, plan, *systems[1][:3]) == 0
    finally:
        dm.dm_destroy(plan)


@pytest.mark.parametrize("m", [72, 100])
def test_conditioned_blocks_keep_digit_products(dm, m):  # noqa: F811
    """Dense blocks of condition 1e4 are graded by 2^8 or so; that is not ambiguous."""
    s = w.conditioned_system(12, m, 1, m, cond=1e4)
    plan = dm.dm_plan(12, m, 1, 3, 1, "fp64")
    try:
        dm.dm_factor(plan, s.A, s.B, s.C)
        assert panels(dm, plan, s.A, s.B, s.C) > 0
    finally:
        dm.dm_destroy(plan)


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


@pytest.mark.parametrize("m,r,N", [(64, 2, 40), (128, 1, 40), (88, 3, 33), (16, 8, 64), (128, 8, 12)])
def test_refinement_of_scaled_unknowns(dm, m, r, N):  # noqa: F811
    """Refined plans, default residual: unknowns over eight decades to the mixed path's 1e-10 of the largest, each in
    its scale, in as many iterations as with the float64 residual (give or take one)."""
    s = w.dominant_system(N, m, r, m)
    A, B, C, b, q = scaled(s, m, 0, 27)
    ref = o.thomas(s.A, s.B, s.C, s.b)
    iters = []
    for mode in ("auto", "fp64"):
        plan = dm.dm_plan(N, m, r, 3, 1, "fp32")
        try:
            dm.dm_set_residual(plan, mode)
            dm.dm_factor(plan, A, B, C)
            x = np.zeros_like(b)
            dm.dm_solve(plan, b, x)
            iters.append(dm.dm_plan_query(plan)["last_iters"])
        finally:
            dm.dm_destroy(plan)
        assert np.max(np.abs(x * q - ref)) <= 1e-10 * np.max(np.abs(ref)), mode
    assert abs(iters[0] - iters[1]) <= 1


def test_neighbours_in_a_batch_do_not_share_scales(dm):  # noqa: F811
    """Three systems of one block size in one level, each in units of its own, their outer blocks NaN: each comes out
    as it does alone."""
    m = 40
    systems = [w.dominant_system(n, m, 1, 60 + n) for n in (12, 9, 15)]
    parts = []
    for k, s in enumerate(systems):
        f = 2.0 ** (-300 * k)
        A, C = s.A * f, s.C * f
        A[0], C[-1] = np.nan, np.nan
        parts.append((A, s.B * f, C, s.b * f))
    plan = dm.dm_plan_batch([s.N for s in systems], [m] * 3, [1] * 3, "fp64")
    try:
        cat = [np.concatenate([p[i].ravel() for p in parts]) for i in range(4)]
        dm.dm_factor(plan, *cat[:3])
        assert panels(dm, plan, *cat[:3]) > 0
        x = np.zeros_like(cat[3])
        dm.dm_solve(plan, cat[3], x, count=3)
    finally:
        dm.dm_destroy(plan)
    at = 0
    for s in systems:
        xs = x[at:at + s.b.size].reshape(s.b.shape)
        at += s.b.size
        assert o.rel_err(xs, o.thomas(s.A, s.B, s.C, s.b)) <= 1e-12
