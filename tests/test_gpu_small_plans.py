"""The one-block launch that plans list offsets for small batches, on either side of its line: offsets are the running sums of the nodes per
query and layer, and a budget out of range is reported."""
import numpy as np
import pytest

from test_gpu_parity import custom_workload

pytestmark = pytest.mark.gpu


def nodes(bp, n):
    return np.clip((bp.astype(np.int64) * n + 5000) // 10000, 1, n)


@pytest.mark.parametrize("n", [1, 2, 1023, 1025, 3071, 3072, 3073, 5000])   # two layers: 6144 entries is the line
@pytest.mark.parametrize("path", ["staged", "fused"])
def test_offsets_are_running_sums(n, path):
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(940, [16, 40, 72, 5], [1, 1, 0], "f32", n=n, n_cal=50, K=2, L=2, budgets=(1, 777, 2500, 9999, 10000))
    dm = harness.DeviceModel(wl)
    g = harness.run_once(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED if path == "staged" else sl.PATH_FUSED)
    per = np.stack([nodes(wl.budget_bp, 40), nodes(wl.budget_bp, 72)], axis=1).reshape(-1)
    assert np.array_equal(g["active_indptr"].astype(np.int64), np.concatenate([[0], np.cumsum(per)]))
    dm.free()


@pytest.mark.parametrize("n", [1000, 3073])
def test_a_budget_out_of_range_is_reported(n):
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(941, [16, 40, 72, 5], [1, 1, 0], "f32", n=n, n_cal=50, K=2, L=2, budgets=(2500,))
    dm = harness.DeviceModel(wl)
    wl.budget_bp[n - 7] = 2501
    b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, max_budget_bp=2500, kernel_path=sl.PATH_STAGED)
    b.run()
    status = b.results()["status"]
    assert int(status[0]) == 5 and int(status[1]) == n - 7
    dm.free()
