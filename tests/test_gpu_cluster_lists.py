"""The one-cluster-per-query path whose list-fed layers run input-stationary, against the oracle: shares of the 16 blocks below and
above one pass of a warp's lanes, empty shares, every number of list positions per thread its selection is compiled for, tables
whose number does not divide the block, inputs that are all zero, plain layers, and a budgeted last layer.  Its selection, which the
layers of tens of queries share, on saved lists that no build writes: against the row kernels."""
import numpy as np
import pytest

from oracle import oracle as orc
from parity_util import assert_run_parity, oracle_model, oracle_run
from test_gpu_parity import custom_workload

pytestmark = pytest.mark.gpu

CASES = {
    # 1024 nodes at 1 to 20 %: 10 to 205 nodes on 16 blocks
    "narrowest": dict(dims=[1024, 1024, 1024, 40], act=[1, 1, 0], dtype="bf16", n=4, budgets=(1, 100, 700, 2000)),
    "ragged": dict(dims=[520, 1160, 1032, 596], act=[1, 1, 1], dtype="f32", n=2, budgets=(300, 2000), K=7, L=3),
    "plain_between": dict(dims=[264, 1416, 1048, 1096, 77], act=[1, 0, 1, 0], dtype="bf16", n=3, budgets=(50, 1900), free_hash=True),
    "more_than_a_pass": dict(dims=[64, 8192, 1024, 16], act=[1, 1, 0], dtype="bf16", n=1, budgets=(2000,)),   # 3276 positions, 1638 inputs
    "a_pass_and_a_bit": dict(dims=[64, 1024, 3072, 333], act=[1, 1, 0], dtype="f32", n=2, budgets=(1700, 2000)),  # 33 and 39 nodes per block
    "eight_tables": dict(dims=[128, 1024, 1400, 50], act=[1, 1, 1], dtype="f32", n=2, budgets=(900, 2000), K=4, L=8),
    "short_lists": dict(dims=[128, 1024, 1024, 10], act=[1, 1, 0], dtype="bf16", n=3, budgets=(200, 2000), list_cap=205, free_hash=True),
    "tiny_layers": dict(dims=[64, 1024, 48, 1024, 24], act=[1, 1, 1, 1], dtype="bf16", n=4, budgets=(1, 400, 2000), K=3, L=2),
}


@pytest.mark.parametrize("name", CASES)
@pytest.mark.parametrize("dead", [False, True])
def test_input_stationary_clusters_match_the_oracle(name, dead):
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    c = CASES[name]
    wl = custom_workload(910, c["dims"], c["act"], c["dtype"], n=c["n"], n_cal=300, K=c.get("K", 10), L=c.get("L", 2), budgets=c["budgets"],
                         list_cap=c.get("list_cap", 0))
    wl.budget_bp[:] = np.resize(c["budgets"], c["n"])
    wl.free_hash_nodes = c.get("free_hash", False)
    if dead:  # the first layer hands over nothing but zeros
        wl.bias[0][:] = -1e4
    dm, om = harness.DeviceModel(wl), oracle_model(wl)
    o32, o64 = (oracle_run(om, wl, wl.x, wl.budget_bp, mode) for mode in (orc.CANON32, orc.REF64))
    for flags, cols in ((0, 10000), (sl.FLAG_ROW_KERNELS, 0)):
        b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_CLUSTER, flags=flags)
        recs = sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes)
        assert [(r["stage"], r["cols_bp"]) for r in recs] == [("cluster", cols)]
        assert acc.kernel_name(acc.NetShape.of(wl), recs[0]) == ("cluster_lists_kernel" if cols else "cluster_network_kernel")
        for _ in range(2):  # again on the same buffers
            b.run()
            assert_run_parity(b.results(), o32, o64, wl, sum(wl.has_act), bool(wl.has_act[-1]))
    lean = harness.DeviceBatch(dm, wl.x, wl.budget_bp, full_outputs=False)
    lean.run()
    assert np.array_equal(lean.results()["pred"], o32["pred"])
    dm.free()


def test_higher_budgets_and_narrow_networks_keep_whole_rows():
    from paper_2204_08400_b200 import binding as sl, harness
    for dims, bp, cols in (([64, 1024, 1024, 10], 2000, 10000), ([64, 1024, 1024, 10], 2001, 0), ([64, 1016, 1016, 10], 2000, 0)):
        wl = custom_workload(911, dims, [1, 1, 0], "bf16", n=2, n_cal=64, K=4, L=2, budgets=(bp,))
        dm = harness.DeviceModel(wl)
        b = harness.DeviceBatch(dm, wl.x, wl.budget_bp)
        assert [r["cols_bp"] for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes) if r["stage"] == "cluster"] == [cols]
        dm.free()


def edited(blob, tables, hash_nodes, edit):
    """A saved model whose bucket lists edit(lists [L, buckets, cap], hash nodes) has changed, with the checksum of its bytes."""
    out, at = blob.copy(), len(blob) - 8
    for t, nodes in zip(reversed(tables), reversed(hash_nodes)):   # layer records end with the lists, the last one at the checksum
        at -= t.nbytes
        edit(out[at:at + t.nbytes].view(t.dtype).reshape(t.shape), nodes.reshape(-1))
        at -= 8 + 4 * nodes.size
    h = 0xCBF29CE484222325
    for b in out[:-8].tobytes():
        h = ((h ^ b) * 0x100000001B3) & 0xFFFFFFFFFFFFFFFF
    out[-8:] = np.frombuffer(h.to_bytes(8, "little"), np.uint8)
    return out


def fill(lists, nodes):
    """Lists that share few nodes, hash nodes left out."""
    others = np.setdiff1d(np.arange(1024), nodes)
    L, buckets, cap = lists.shape
    b, k, r = np.ogrid[:L, :buckets, :cap]
    lists[...] = others[(b * 450 + k * 13 + r) % others.size]


def name_a_hash_node(lists, nodes):
    fill(lists, nodes)
    lists[:, :, 0] = nodes[1]


def name_three_hash_nodes(lists, nodes):
    fill(lists, nodes)
    lists[:, :, (0, 5, 9)] = nodes[:3]


def one_node_only(lists, nodes):
    lists[...] = np.setdiff1d(np.arange(1024), nodes)[700]


@pytest.mark.parametrize("edit,short", [(name_a_hash_node, False), (name_three_hash_nodes, False), (one_node_only, True)])
@pytest.mark.parametrize("path,n,kernel", [("CLUSTER", 3, "cluster_lists_kernel"), ("STAGED", 80, "few_nodes_kernel")])
def test_saved_lists_that_name_hash_nodes(edit, short, path, n, kernel):
    """Loading checks the sizes and the checksum of the lists, not their entries.  An entry that names an always-active hash node
    is not counted, and a query whose lists are too short is reported and takes the first nodes, as in the row kernels."""
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    wl = custom_workload(912, [64, 1024, 1024, 40], [1, 1, 0], "bf16", n=n, n_cal=200, K=4, L=2, budgets=(200, 1000, 2000), list_cap=300)
    wl.free_hash_nodes = True
    dm = harness.DeviceModel(wl)
    blob = sl.slonn_serialize(dm.model)
    assert np.array_equal(edited(blob, [dm.tables(0), dm.tables(1)], [dm.hash_nodes(0), dm.hash_nodes(1)], lambda lists, nodes: None), blob)
    blob = edited(blob, [dm.tables(0), dm.tables(1)], [dm.hash_nodes(0), dm.hash_nodes(1)], edit)
    built, dm.model = dm.model, sl.slonn_deserialize(blob, dm.W, dm.bias)
    got = []
    for flags in (0, sl.FLAG_ROW_KERNELS):
        b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=getattr(sl, "PATH_" + path), flags=flags)
        names = [acc.kernel_name(acc.NetShape.of(wl), r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes)]
        assert (kernel in names) == (flags == 0)
        got.append(b.results())
    assert [bool(g["status"][0]) for g in got] == [short, short] and (not short or got[0]["status"][0] == -sl.ERR["ARG"])
    for k in ("logits", "pred", "codes", "active_indptr", "active_ids", "active_vals"):
        assert np.array_equal(got[0][k], got[1][k]), k
    sl.slonn_free(built)
    dm.free()
