"""A plan with float32 factors and m % 8 != 0 whose supplementary levels' digit slices do not fit the free memory is
planned without them, as a float64 plan is: what fitted on the float64 pipe still fits."""
import numpy as np
import pytest

from paper_1505_06864_gb300 import workloads as w
from test_gpu_blocked_inverse import dm  # noqa: F401

pytestmark = pytest.mark.gpu


def test_refined_plan_without_room_for_slices(dm):  # noqa: F811
    import torch
    N, m, P = 2401, 100, 1200

    def plan_bytes():
        plan = dm.dm_plan(N, m, 1, P, 1, "fp32")
        try:
            return dm.dm_plan_query(plan)["device_bytes"]
        finally:
            dm.dm_destroy(plan)

    sliced = plan_bytes()
    slices = 3 * 7 * m * 104 * 2 * (P - 1)  # of A, C and Acal: seven bf16 digits, rows padded to 104
    assert sliced > 2 * slices
    free, _ = torch.cuda.mem_get_info()
    hold = torch.empty(free - (1 << 30) - sliced + slices // 2, dtype=torch.uint8, device="cuda")  # 1 GB: the reserve
    try:
        assert plan_bytes() < sliced - slices
    finally:
        del hold
        torch.cuda.empty_cache()
    s = w.dominant_system(9, m, 1, 5)  # and with room again the slices are back
    plan = dm.dm_plan(9, m, 1, 3, 1, "fp32")
    try:
        dm.dm_factor(plan, s.A, s.B, s.C)
        x = np.zeros_like(s.b)
        dm.dm_solve(plan, s.b, x)
    finally:
        dm.dm_destroy(plan)
    assert plan_bytes() == sliced
    assert np.max(np.abs(x - s.x_true)) <= 1e-10 * np.max(np.abs(s.x_true))
