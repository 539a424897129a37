"""List-fed layers of batches of tens of queries (few_select_kernel, few_nodes_kernel) against the oracle: last runs of four columns and
last blocks half full, more queries than SMs, every number of list positions per thread, tables whose number does not divide
a block, budgets that differ, inputs that are all zero, infinities and NaNs, plain layers in the middle and at the end; a workspace
without their scratch, a saved model, and queries from host memory."""
import numpy as np
import pytest

from oracle import oracle as orc
from parity_util import assert_run_parity, oracle_model, oracle_run
from test_gpu_parity import custom_workload

pytestmark = pytest.mark.gpu

CASES = {
    "smallest": dict(dims=[64, 1024, 1024, 36], act=[1, 1, 0], dtype="bf16", n=80, budgets=(1, 100, 5000)),
    "ragged": dict(dims=[136, 1160, 1036, 596], act=[1, 1, 1], dtype="f32", n=97, budgets=(300, 2000, 4900), K=7, L=3),
    "more_queries_than_sms": dict(dims=[64, 1032, 1304, 44], act=[1, 1, 0], dtype="bf16", n=173, budgets=(1000, 2500)),
    "widest": dict(dims=[32, 8192, 8192, 20], act=[1, 1, 0], dtype="bf16", n=40, budgets=(2000, 2500)),       # 4096 list positions
    "eight_tables": dict(dims=[64, 2048, 1400, 52], act=[1, 1, 1], dtype="f32", n=41, budgets=(900, 3600), K=4, L=8),
    "short_lists": dict(dims=[64, 2056, 1024, 12], act=[1, 1, 0], dtype="bf16", n=40, budgets=(200, 2000), list_cap=430, free_hash=True),
    # layers without activator: the last block of runs a third full, the last run of columns the only one of its block
    "plain_last": dict(dims=[64, 1024, 1024, 1036], act=[1, 1, 0], dtype="bf16", n=64, budgets=(300, 1000, 1500), plain=2),
    "plain_last_f32": dict(dims=[64, 1028, 1024, 772], act=[1, 1, 0], dtype="f32", n=65, budgets=(1, 900, 1500), K=7, L=3, plain=2),
    "plain_between": dict(dims=[64, 1024, 1032, 1032, 72], act=[1, 1, 0, 0], dtype="bf16", n=80, budgets=(200, 2000), free_hash=True, list_cap=300, plain=2),
    "plain_between_f32": dict(dims=[64, 1024, 1024, 900, 1028, 24], act=[1, 1, 0, 1, 0], dtype="f32", n=96, budgets=(500, 3500), plain=2),
    "small_layer": dict(dims=[64, 1024, 120, 24], act=[1, 1, 1], dtype="bf16", n=81, budgets=(1, 400, 5000), K=3, L=2),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("dead", [False, True])
def test_layers_of_few_queries_match_the_oracle(name, dead):
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    c = CASES[name]
    wl = custom_workload(930, c["dims"], c["act"], c["dtype"], n=c["n"], n_cal=200, K=c.get("K", 10), L=c.get("L", 2), budgets=c["budgets"],
                         list_cap=c.get("list_cap", 0))
    wl.budget_bp[:] = np.resize(c["budgets"], c["n"])
    wl.free_hash_nodes = c.get("free_hash", False)
    if dead:  # the first layer hands over nothing but zeros
        wl.bias[0][:] = -1e4
    dm, om = harness.DeviceModel(wl), oracle_model(wl)
    o32, o64 = (oracle_run(om, wl, wl.x, wl.budget_bp, mode) for mode in (orc.CANON32, orc.REF64))
    b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED)
    names = [acc.kernel_name(acc.NetShape.of(wl), r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes) if r["layer"] == 1]
    assert names == ["few_select_kernel", "few_nodes_kernel"]
    if "plain" in c:
        names = [acc.kernel_name(acc.NetShape.of(wl), r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes) if r["layer"] == c["plain"]]
        assert names == ["few_nodes_kernel"]
    for _ in range(2):
        b.run()
        assert_run_parity(b.results(), o32, o64, wl, sum(wl.has_act), bool(wl.has_act[-1]))
    # a workspace of the size the other kernels need: those run, with the same results
    least = sl.slonn_workspace_bytes(dm.model, b.n, b.max_bp, sl.FLAG_ROW_KERNELS)
    assert least < b.ws_bytes
    sl.slonn_run(dm.model, b.batch, b.ws, least)
    assert_run_parity(b.results(), o32, o64, wl, sum(wl.has_act), bool(wl.has_act[-1]))
    names = [acc.kernel_name(acc.NetShape.of(wl), r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, least) if r["layer"] == 1]
    assert "few_nodes_kernel" not in names
    dm.free()


def test_lines_of_the_dispatch():
    """Queries times inputs, nodes per query, largest budget: both sides of each line."""
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    for dims, n, bp, few in (([64, 1024, 1024, 8], 80, 1501, True), ([64, 1024, 1024, 8], 79, 1501, False), ([64, 1024, 1024, 8], 48, 1000, True), ([64, 1024, 1024, 8], 47, 1000, False), ([64, 1024, 1024, 8], 48, 500, False),
                             ([64, 1024, 1024, 8], 150, 1000, True), ([64, 2048, 2048, 8], 150, 600, False), ([64, 2048, 2048, 8], 150, 700, True),
                             # more than 1640 nodes: 40 queries
                             ([64, 4096, 4096, 8], 39, 4000, True), ([64, 4096, 4096, 8], 39, 4100, False), ([64, 4096, 4096, 8], 40, 4100, True),
                             # fp32, 2048 inputs and more: layer_cols_kernel keeps 9472 nodes of a batch and more, up to 215 a query and 128 queries
                             ([64, 2048, 2052, 8], 80, 1000, False), ([64, 2048, 2052, 8], 80, 1100, True), ([64, 2048, 2052, 8], 46, 1000, True),
                             ([64, 2048, 2052, 8], 128, 1000, False), ([64, 2048, 2052, 8], 129, 1000, True),
                             ([64, 1024, 1022, 8], 90, 2500, False), ([64, 1024, 1024, 8], 90, 5001, False)):
        wl = custom_workload(931, dims, [1, 1, 0], "f32" if dims[2] % 8 else "bf16", n=n, n_cal=64, K=4, L=2, budgets=(bp,)) if dims[2] % 4 == 0 else \
            custom_workload(931, dims[:2] + [dims[2]], [1, 1], "bf16", n=n, n_cal=64, K=4, L=2, budgets=(bp,))
        dm = harness.DeviceModel(wl)
        b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED)
        names = [acc.kernel_name(acc.NetShape.of(wl), r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes) if r["layer"] == 1]
        assert ("few_nodes_kernel" in names) == few, (dims, n, bp, names)
        dm.free()


@pytest.mark.parametrize("n,few", [(255, True), (256, False), (700, False)])
def test_batches_that_may_not_group_queries(n, few):
    """Without grouped products these kernels would be all that is left of the forms with scratch: they end below 256 queries, and so
    does their scratch."""
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    wl = custom_workload(932, [64, 1024, 1024, 8], [1, 1, 0], "bf16", n=n, n_cal=64, K=4, L=2, budgets=(2500,))
    dm = harness.DeviceModel(wl)
    b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED, flags=sl.FLAG_UNGROUPED_ROWS)
    names = [acc.kernel_name(acc.NetShape.of(wl), r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes) if r["layer"] == 1]
    assert ("few_nodes_kernel" in names) == few, names
    assert (b.ws_bytes > sl.slonn_workspace_bytes(dm.model, n, 2500, sl.FLAG_ROW_KERNELS)) == few
    got = b.results()
    rows = harness.run_once(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED, flags=sl.FLAG_ROW_KERNELS | sl.FLAG_UNGROUPED_ROWS)
    for k in ("logits", "pred", "codes", "active_indptr", "active_ids", "active_vals"):
        assert np.array_equal(got[k], rows[k]), k
    dm.free()


@pytest.mark.parametrize("n,last,few", [(48, 1024, True), (48, 1020, False), (64, 768, True), (64, 764, False)])
def test_lines_of_plain_layers(n, last, few):
    """Queries times outputs: 48 K."""
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    wl = custom_workload(933, [64, 1024, 1024, last], [1, 1, 0], "bf16", n=n, n_cal=64, K=4, L=2, budgets=(1000,))
    dm = harness.DeviceModel(wl)
    b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED)
    names = [acc.kernel_name(acc.NetShape.of(wl), r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes) if r["layer"] == 2]
    assert ("few_nodes_kernel" in names) == few, names
    dm.free()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("path,n", [("CLUSTER", 4), ("STAGED", 64)])
def test_infinities_and_nans(dtype, path, n):
    """Infinite and NaN inputs give what the row kernels give, and leave the other queries of the batch alone."""
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(934, [64, 1024, 1032, 1036], [1, 1, 0], dtype, n=n, n_cal=200, K=6, L=2, budgets=(300, 1500))
    w = wl.W_store[1]   # every other node of the second layer adds up positive weights, so that infinities stay infinities
    w[::2] = np.abs(w[::2]) if dtype == "f32" else w[::2] & 0x7FFF
    dm = harness.DeviceModel(wl)
    x = wl.x.copy()
    x[1::4, 3], x[2::4, 9], x[2::4, 11] = np.inf, np.nan, -np.inf
    clean, dirty = (harness.run_once(dm, v, wl.budget_bp, kernel_path=getattr(sl, "PATH_" + path)) for v in (wl.x, x))
    rows = harness.run_once(dm, x, wl.budget_bp, kernel_path=getattr(sl, "PATH_" + path), flags=sl.FLAG_ROW_KERNELS)
    assert np.isinf(dirty["active_vals"]).any() and np.isnan(dirty["logits"][1::4]).any()
    for k in ("logits", "pred", "codes", "active_indptr", "active_ids", "active_vals"):
        assert np.array_equal(dirty[k], rows[k], equal_nan=dirty[k].dtype == np.float32), k
    others = [q for q in range(n) if q % 4 in (0, 3)]
    assert np.array_equal(clean["logits"][others], dirty["logits"][others])
    dm.free()


@pytest.mark.parametrize("n,kernel", [(3, "cluster_lists_kernel"), (64, "few_nodes_kernel")])
def test_saved_models_and_host_buffers(n, kernel):
    """The copies these kernels read are made again on loading; queries in host memory take the same kernels in the call's own workspace."""
    import torch
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    wl = custom_workload(935, [64, 1024, 1040, 1020], [1, 1, 0], "bf16", n=n, n_cal=200, K=6, L=2, budgets=(400, 1500))
    dm = harness.DeviceModel(wl)
    want = harness.run_once(dm, wl.x, wl.budget_bp)
    built, dm.model = dm.model, sl.slonn_deserialize(sl.slonn_serialize(dm.model), dm.W, dm.bias)
    sl.slonn_free(built)
    b = harness.DeviceBatch(dm, wl.x, wl.budget_bp)
    assert kernel in [acc.kernel_name(acc.NetShape.of(wl), r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes)]
    b.run()
    got = b.results()
    for k in ("logits", "pred", "codes", "active_indptr", "active_ids", "active_vals"):
        assert np.array_equal(got[k], want[k]), k
    full = sl.slonn_host_workspace_bytes(dm.model, n, 1500)
    least = sl.slonn_host_workspace_bytes(dm.model, n, 1500, flags=sl.FLAG_ROW_KERNELS)
    for nb in {full, least}: # with and without scratch
        logits, pred, status = np.zeros((n, 1020), np.float32), np.zeros(n, np.uint32), np.ones(4, np.uint32)
        hb = sl.make_batch(n, np.ascontiguousarray(wl.budget_bp), logits, status, x_dense=np.ascontiguousarray(wl.x), max_budget_bp=1500, pred=pred)
        sl.slonn_run_host(dm.model, hb, torch.empty(nb, dtype=torch.uint8, device=dm.device), nb)
        assert status[0] == 0
        assert np.array_equal(logits, want["logits"]) and np.array_equal(pred, want["pred"])
    dm.free()
