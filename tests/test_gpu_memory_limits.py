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
