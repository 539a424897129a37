"""Runs queued back to back on changing inputs in the same buffers: a kernel that read what the one before it was still
writing would return parts of an earlier batch."""
import numpy as np
import pytest

from test_gpu_parity import check, custom_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,has_act,n", [
    ([512, 640, 1032, 768, 520, 24], [0, 0, 0, 1, 0], 320),     # three plain layers in a row, then a list-fed one
    ([512, 640, 1032, 768, 520, 24], [0, 0, 0, 1, 0], 16),      # the same with the kernels for tens of queries
    ([256, 1536, 1536, 640], [0, 0, 1], 520),                   # two plain layers in front of a budgeted output
])
def test_plain_layers_in_a_row_on_changing_inputs(dims, has_act, n):
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(4300 + n, dims, has_act, "bf16", n=n, n_cal=300, K=4, L=2, budgets=(700, 3000, 5000))
    check(wl)
    dm = harness.DeviceModel(wl)
    b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED)
    xs = [b.x_dense.clone(), b.x_dense.flip(0).contiguous(), b.x_dense * 0.5]
    want = []
    for x in xs:
        b.x_dense.copy_(x)
        b.run()
        want.append(b.results())
    for turn in range(12):   # nobody waits between the runs; the last one's results are looked at
        for i in (0, 1, 2, turn % 3):
            b.x_dense.copy_(xs[i])
            b.run()
        got = b.results()
        for k in ("logits", "pred", "codes", "active_ids", "active_vals"):
            assert np.array_equal(got[k], want[turn % 3][k]), (turn, k)
    dm.free()


def test_csr_fed_first_layer_on_changing_inputs():
    from paper_2204_08400_b200 import binding as sl, harness, workloads as wl_mod
    wl = wl_mod.load("c3", n_queries=300, n_cal=300, budget_bp=1000, dims=[4000, 128, 3000])
    check(wl)
    dm = harness.DeviceModel(wl)
    b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED)
    vals = b.x_csr[2]
    vs = [vals.clone(), vals.flip(0).contiguous(), vals * 0.5]
    want = []
    for v in vs:
        vals.copy_(v)
        b.run()
        want.append(b.results())
    for turn in range(12):
        for i in (0, 1, 2, turn % 3):
            vals.copy_(vs[i])
            b.run()
        got = b.results()
        for k in ("logits", "pred", "codes", "active_ids", "active_vals"):
            assert np.array_equal(got[k], want[turn % 3][k]), (turn, k)
    dm.free()


def test_two_threads_with_a_stream_each():
    """One model, two host threads, two streams, batches of different sizes and budgets that take the grouped products, each
    with a workspace of its own: every run's results are those of the batch alone."""
    import threading
    import torch
    from paper_2204_08400_b200 import harness
    wl = custom_workload(4350, [512, 1536, 1536, 130], [1, 1, 0], "bf16", n=700, n_cal=300, K=4, L=2,
                         budgets=(1000, 5000, 9000, 10000))
    dm = harness.DeviceModel(wl)
    parts = [(wl.x, wl.budget_bp), (wl.x[:300], np.full(300, 6000, np.uint16))]
    batches = [harness.DeviceBatch(dm, x, bp, kernel_path=1) for x, bp in parts]
    want = []
    for b in batches:
        b.run()
        want.append(b.results())
    streams = [torch.cuda.Stream() for _ in parts]
    torch.cuda.synchronize()
    keys = ("logits", "pred", "codes", "active_ids", "active_vals")
    wrong = []

    def work(i):
        for _ in range(15):
            for t in (batches[i].logits, batches[i].vals, batches[i].ids):
                with torch.cuda.stream(streams[i]):
                    t.zero_()
            batches[i].run(streams[i])
            batches[i].run(streams[i])
            streams[i].synchronize()
            got = batches[i].results()
            wrong.extend((i, k) for k in keys if not np.array_equal(got[k], want[i][k]))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong[:4]
    dm.free()
