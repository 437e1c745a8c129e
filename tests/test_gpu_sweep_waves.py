"""Solve sweeps of subsystems with different block sizes in more waves of clusters than are resident together (eight
CTAs to a cluster at m = 256, so 36 to 148 of them): float64 and refined float32 factors, few and many right-hand
sides.  Tolerances: the paths' 1e-12 and 1e-10 of the oracle on dominant systems."""
import numpy as np
import pytest

from oracle import dm_oracle as o
from paper_1505_06864_gb300 import workloads as w
from test_gpu_blocked_inverse import dm  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPES = [(150, 24, 1), (64, 256, 2), (130, 72, 3), (33, 160, 1), (200, 33, 2), (120, 64, 1)]


@pytest.mark.parametrize("r", [1, 16])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-10)])
def test_mixed_sizes(dm, prec, tol, r):  # noqa: F811
    shapes = [(n, m, max(1, q * r // 2)) for n, m, q in SHAPES] if r == 1 else [(n, m, r) for n, m, _ in SHAPES]
    systems = [w.dominant_system(n, m, q, 40 + k) for k, (n, m, q) in enumerate(shapes)]
    plan = dm.dm_plan_batch(*[list(v) for v in zip(*shapes)], prec)
    try:
        cat = lambda f: np.concatenate([f(s).ravel() for s in systems])  # noqa: E731
        dm.dm_factor(plan, cat(lambda s: s.A), cat(lambda s: s.B), cat(lambda s: s.C))
        x = np.zeros(sum(s.b.size for s in systems))
        dm.dm_solve(plan, cat(lambda s: s.b), x, count=len(shapes))
    finally:
        dm.dm_destroy(plan)
    at = 0
    for s in systems:
        xs = x[at:at + s.b.size].reshape(s.b.shape)
        at += s.b.size
        assert np.all(np.isfinite(xs))
        assert o.rel_err(xs, o.dm(s.A, s.B, s.C, s.b, 8)) <= tol
