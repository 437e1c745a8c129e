"""The tensor-core residual entry by entry: its error against the sum of the entry's own terms' magnitudes, where those
are far below the largest entries of the row and of x (unknowns of different scale, solutions that decay inside a
block, single unknowns), at the edges of its tiles and column classes.

Bound: 3m 2^-49 sum |row of [A B C]| |column of x|, the largest that the digit products may have where their entry is
certified (3m 2^-55 of the scales, of which the sum is at least 2^-6), and above the float64 recomputation's."""
import numpy as np
import pytest

from paper_1505_06864_gb300 import workloads as w
from test_gpu_residual import dm, exact_residual  # noqa: F401

pytestmark = pytest.mark.gpu


def magnitudes(s, x):
    S = np.matmul(np.abs(s.B), np.abs(x))
    S[1:] += np.matmul(np.abs(s.A[1:]), np.abs(x[:-1]))
    S[:-1] += np.matmul(np.abs(s.C[:-1]), np.abs(x[1:]))
    return S


def case(kind, N, m, r):
    rng = np.random.default_rng(7 * m + r)
    s = w.pde_banded_system(N, m, r, m) if kind in ("decay", "single") and m >= 8 else w.dominant_system(N, m, r, m)
    x = rng.standard_normal((N, m, r))
    if kind == "scaled":
        q = np.ldexp(1.0, -rng.integers(0, 41, size=(N, m)))
        s.B *= q[:, None, :]
        s.A[1:] *= q[:-1, None, :]
        s.C[:-1] *= q[1:, None, :]
        x /= q[:, :, None]
    elif kind == "decay":
        x *= np.ldexp(1.0, -(np.arange(m) * 60 // m))[None, :, None]
        x[:, :, 0] = x[:, ::-1, 0]
    elif kind == "single":
        x[:] = 0.0
        x[N // 2, m // 2] = rng.standard_normal(r)
        x[0, 0] = 1e-20
    return s, x


@pytest.mark.parametrize("kind", ["plain", "scaled", "decay", "single"])
@pytest.mark.parametrize("N,m,r", [(1, 5, 1), (9, 15, 8), (8, 16, 9), (17, 16, 1), (5, 31, 16), (6, 64, 2), (3, 65, 9),
                                   (3, 128, 8), (2, 127, 16)])
def test_error_against_the_entry_s_own_terms(dm, N, m, r, kind):  # noqa: F811
    s, x = case(kind, N, m, r)
    plan = dm.dm_plan(N, m, r, 1, 1, "fp64")
    try:
        dm.dm_set_residual(plan, "sliced")
        dm.dm_factor(plan, s.A, s.B, s.C)
        b = np.zeros_like(s.b)
        res = np.zeros_like(b)
        dm.dm_residual(plan, x, b, res)
        assert dm.dm_plan_query(plan)["residual_tc_systems"] == 1
    finally:
        dm.dm_destroy(plan)
    err = np.abs(res.astype(np.longdouble) - exact_residual(s.A, s.B, s.C, x, b)).astype(np.float64)
    assert np.all(err <= 3 * m * 2.0 ** -49 * magnitudes(s, x))
