"""Float64 levels with blocks of at most 32 (the whole factor sweep in one launch): every pivot exchanged, sizes
around the warps' column shares (2, 4, 8), mixed sizes in one level, recursion, subsystems of one row, banded
blocks, a singular block.  Tolerance: the float64 path's 1e-12 of the oracle on well-conditioned systems."""
import numpy as np
import pytest

from oracle import dm_oracle as o
from paper_1505_06864_gb300 import workloads as w
from test_gpu_blocked_inverse import dm, permuted_system  # noqa: F401

pytestmark = pytest.mark.gpu

TOL = 1e-12


def check(x, xref):
    assert np.all(np.isfinite(x))
    assert np.all(np.max(np.abs(x - xref), axis=(0, 1)) <= TOL * np.max(np.abs(xref), axis=(0, 1)))
    assert o.rel_err(x, xref) <= TOL


@pytest.mark.parametrize("N,m,r,P,levels", [(1, 1, 1, 1, 1), (7, 2, 1, 4, 1), (9, 7, 1, 2, 1), (20, 8, 2, 5, 2),
                                            (9, 9, 1, 3, 1), (40, 16, 1, 12, 2), (9, 17, 3, 2, 1), (12, 31, 1, 3, 1),
                                            (12, 32, 2, 3, 1)])
def test_every_pivot_exchanged(dm, N, m, r, P, levels):  # noqa: F811
    s = permuted_system(N, m, r, 3 * m + N)
    plan = dm.dm_plan(N, m, r, P, levels, "fp64")
    try:
        dm.dm_factor(plan, s.A, s.B, s.C)
        x = np.zeros_like(s.b)
        dm.dm_solve(plan, s.b, x)
    finally:
        dm.dm_destroy(plan)
    check(x, o.dm(s.A, s.B, s.C, s.b, P))


@pytest.mark.parametrize("m,hb", [(16, 0), (17, 3), (32, 6), (24, 7)])
def test_banded_blocks(dm, m, hb):  # noqa: F811
    s = w.pde_banded_system(30, m, 2, m + hb, hb=hb)
    plan = dm.dm_plan(30, m, 2, 4, 1, "fp64")
    try:
        dm.dm_factor(plan, s.A, s.B, s.C)
        x = np.zeros_like(s.b)
        dm.dm_solve(plan, s.b, x)
    finally:
        dm.dm_destroy(plan)
    check(x, o.dm(s.A, s.B, s.C, s.b, 4))


def test_mixed_sizes_in_one_level(dm):  # noqa: F811
    shapes = [(40, 5, 1), (64, 16, 3), (33, 32, 2), (25, 24, 1)]
    systems = [permuted_system(n, m, r, 90 + k) for k, (n, m, r) in enumerate(shapes)]
    plan = dm.dm_plan_batch(*[list(v) for v in zip(*shapes)], "fp64")
    try:
        cat = lambda f: np.concatenate([f(s).ravel() for s in systems])  # noqa: E731
        dm.dm_factor(plan, cat(lambda s: s.A), cat(lambda s: s.B), cat(lambda s: s.C))
        x = np.zeros(sum(s.b.size for s in systems))
        dm.dm_solve(plan, cat(lambda s: s.b), x, count=len(shapes))
    finally:
        dm.dm_destroy(plan)
    off = 0
    for s in systems:
        check(x[off:off + s.b.size].reshape(s.b.shape), o.thomas(s.A, s.B, s.C, s.b))
        off += s.b.size


def test_singular_block(dm):  # noqa: F811
    s = w.dominant_system(12, 16, 1, 4)
    s.B[5] = 0.0
    s.A[5] = 0.0  # row 5 of the block Thomas sweep: D = B - A Acal = 0
    plan = dm.dm_plan(12, 16, 1, 1, 1, "fp64")
    try:
        with pytest.raises(dm.DMError) as e:
            dm.dm_factor(plan, s.A, s.B, s.C)
        assert e.value.code == dm.DM_ESINGULAR and "block row 5" in str(e.value)
    finally:
        dm.dm_destroy(plan)
