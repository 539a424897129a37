"""Calls that use device memory they can do without must work when there is none left."""
import contextlib
import ctypes as C

import numpy as np
import pytest

from test_gpu_parity import custom_workload

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def memory_taken(leave):
    """All of the GPU's free memory but `leave` bytes (0: until 256 KB cannot be had) is held while the block runs."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    cu = C.CDLL("libcuda.so.1")
    held = []
    try:
        step = 8 << 30
        while step >= 256 << 10:
            p = C.c_uint64()
            fits = leave == 0 or torch.cuda.mem_get_info()[0] >= leave + step
            if fits and cu.cuMemAlloc_v2(C.byref(p), C.c_size_t(step)) == 0:
                held.append(p)
            else:
                step //= 2
        yield
    finally:
        for p in held:
            cu.cuMemFree_v2(p)


def test_a_first_layer_without_room_for_its_copy_still_builds():
    """8192 x 16384 fp32: the copy takes 512 MB, 300 are left (calibration and tables take 20)."""
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(4600, [8192, 16384, 16], [1, 0], "f32", n=300, n_cal=64, K=2, L=1, budgets=(300, 10000))
    dm = harness.DeviceModel(wl)
    want = harness.run_once(dm, wl.x, wl.budget_bp)
    dm.free()
    dm2 = harness.DeviceModel.__new__(harness.DeviceModel)
    dm2.wl, dm2.device, dm2.W, dm2.bias = wl, dm.device, dm.W, dm.bias
    import torch
    calib = torch.from_numpy(wl.calib).cuda()
    with memory_taken(300 << 20):
        dm2.model = sl.slonn_build(wl.dims, wl.has_act, sl.SLONN_F32, dm2.W, dm2.bias, calib_dense=calib, K=wl.K, L=wl.L,
                                   list_cap=wl.list_cap, seed=wl.seed)
    got = harness.run_once(dm2, wl.x, wl.budget_bp)   # 100 % queries among them: the row kernels compute their first layer
    for k in ("logits", "pred", "codes", "active_ids", "active_vals"):
        assert np.array_equal(got[k], want[k]), k
    dm2.free()


def test_the_first_layers_copy_carries_nothing_nobody_reads():
    """A dense first layer of 57,344 inputs: its side-by-side hash rows would take 7.4 MB beside its copy (7.4 MB) and tables."""
    import torch
    from paper_2204_08400_b200 import harness
    wl = custom_workload(4601, [57344, 32, 16], [1, 0], "f32", n=8, n_cal=64, K=2, L=1)
    harness.DeviceModel(wl).free()                    # kernels and pools are in place from here on
    dm = harness.DeviceModel(wl)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    dm.free()
    torch.cuda.synchronize()
    held = torch.cuda.mem_get_info()[0] - before
    assert held < (57344 * 32 * 4) + (6 << 20), held  # the copy, and a few pieces of 2 MB each


def test_saving_needs_no_device_memory():
    """4 MB of tables: their checksum is taken on the device when its scratch can be had, else on the host."""
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(4602, [64, 1028, 8], [1, 0], "f32", n=8, n_cal=300, K=10, L=2)
    dm = harness.DeviceModel(wl)
    blob = sl.slonn_serialize(dm.model)
    with memory_taken(0):
        again = sl.slonn_serialize(dm.model)
    assert np.array_equal(again, blob)
    dm.free()
