"""Layers evaluated as grouped products (16 queries x 128 or 256 columns per work item): sizes at the edges of a tile, a group, a
partial sum's stretch and a staged chunk, against the oracle or bit for bit against the row kernels (whose own parity the
other tests cover; the order of every sum is fixed, so the two have to agree in every bit)."""
import numpy as np
import pytest

from test_gpu_parity import check, custom_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,dims,has_act,n,budgets", [
    ("bf16", [264, 128, 136, 127], [1, 1, 1], 256, (3600, 5000, 9999)),         # one tile, one tile and 8 columns, odd width
    ("f32", [132, 260, 124, 61], [1, 1, 0], 273, (4000, 7500, 10000)),          # ragged last group, odd output layer
    ("bf16", [8, 32, 40, 3], [1, 1, 0], 259, (9000, 10000)),                    # partial sums without any input
    ("f32", [64, 1032, 1024, 130], [1, 1, 1], 300, (300, 3499, 3501, 6000)),    # both sides of the split with layer_cols
])
def test_grouped_products_at_the_edges_of_their_tiles(dtype, dims, has_act, n, budgets):
    wl = custom_workload(4100 + n, dims, has_act, dtype, n=n, n_cal=300, K=4, L=2, budgets=budgets)
    check(wl)


def _run(dm, wl, flags=0, ws_bytes=None, x=None):
    from paper_2204_08400_b200 import binding as sl, harness
    b = harness.DeviceBatch(dm, wl.x if x is None else x, wl.budget_bp, kernel_path=sl.PATH_STAGED, flags=flags)
    if ws_bytes is not None:
        b.ws_bytes = ws_bytes
    b.run()
    return b.results()


KEYS = ("logits", "pred", "codes", "active_ids", "active_vals")


def _same_bits(a, b):
    for k in KEYS:
        assert np.array_equal(a[k].view(np.uint8), b[k].view(np.uint8)), k


def test_grouped_products_in_several_chunks():
    """More queries than are sorted and staged at a time (8192), 100 % queries among them."""
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(4201, [64, 600, 520, 20], [1, 1, 0], "bf16", n=8192 + 8192 + 17, n_cal=300, K=4, L=2,
                         budgets=(1000, 5000, 10000))
    dm = harness.DeviceModel(wl)
    _same_bits(_run(dm, wl), _run(dm, wl, flags=sl.FLAG_ROW_KERNELS))
    dm.free()


@pytest.mark.parametrize("dtype,dims,has_act,n,budgets", [
    ("bf16", [40, 264, 256, 250], [1, 0, 0], 1209, (5000,)),              # every node: one item of exactly 256 columns, one short of it
    ("f32", [36, 264, 252, 253], [1, 0, 0], 1209, (5000,)),
    ("bf16", [8, 248, 256, 505], [1, 1, 0], 2500, (10000,)),              # 100 % queries, two items, the second not full
    ("bf16", [1032, 520, 528, 24], [1, 1, 0], 8209, (4850, 4880, 9999)),  # selected nodes, up to one more than an item holds
    ("f32", [132, 516, 260, 24], [1, 1, 0], 8192, (9000, 9900)),
])
def test_layers_of_up_to_256_columns_and_more(dtype, dims, has_act, n, budgets):
    """Around the 256 columns of the longer work items, whichever kernel takes them; partial sums without an input and odd widths among
    them.  (test_which_product_kernel_is_taken and test_item_width_follows_the_queries_that_are_served ask for the kernel too.)"""
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(4300 + n, dims, has_act, dtype, n=n, n_cal=300, K=4, L=2, budgets=budgets)
    dm = harness.DeviceModel(wl)
    _same_bits(_run(dm, wl), _run(dm, wl, flags=sl.FLAG_ROW_KERNELS | sl.FLAG_UNGROUPED_ROWS))
    dm.free()


@pytest.mark.parametrize("dtype,n,last", [("bf16", 40, 505), ("f32", 33, 576), ("bf16", 200, 500), ("f32", 255, 641), ("bf16", 64, 296)])
def test_plain_layers_of_few_queries_by_input(dtype, n, last):
    """A layer without activator behind a list of 2048 inputs: odd widths, a last block that is not full.  (The form is asked for in
    test_plain_layers_of_few_queries_take_columns_where_they_pay.)"""
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(4700 + n, [64, 2048, last], [1, 0], dtype, n=n, n_cal=200, K=4, L=2, budgets=(20, 2000, 3500))
    dm = harness.DeviceModel(wl)
    _same_bits(_run(dm, wl), _run(dm, wl, flags=sl.FLAG_ROW_KERNELS | sl.FLAG_UNGROUPED_ROWS))
    dm.free()


@pytest.mark.parametrize("dtype,n,last,kernel", [
    ("bf16", 2000, 10, "gather_dot_kernel"),    # a block's 64 nodes are mostly padding
    ("bf16", 37, 512, "gather_dot_kernel"),     # 18,944 rows; from 23,680 on
    ("f32", 47, 504, "gather_cols_kernel"),
    ("bf16", 493, 48, "gather_dot_kernel"),     # 23,664
    ("bf16", 494, 48, "gather_cols_kernel"),
    ("bf16", 750, 200, "gather_dot_kernel"),    # 3000 blocks; below 2368
    ("f32", 592, 200, "gather_dot_kernel"),
    ("f32", 591, 200, "gather_cols_kernel"),
    ("bf16", 215, 641, "gather_cols_kernel"),   # an odd width, 2365 blocks
    ("bf16", 255, 641, "gather_cols_kernel"),   # as many rows as fill the GPU: whole queries per block
])
def test_plain_layers_of_few_queries_take_columns_where_they_pay(dtype, n, last, kernel):
    """Both sides of each line of the dispatch, at budgets that smaller batches leave to the row kernels; same bits as these."""
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    wl = custom_workload(4900 + n, [64, 2048, last], [1, 0], dtype, n=n, n_cal=200, K=4, L=2, budgets=(300, 2000, 3500))
    dm = harness.DeviceModel(wl)
    b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED)
    names = [acc.kernel_name(acc.NetShape.of(wl), r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes) if r["layer"] == 1]
    assert names == [kernel], names
    _same_bits(b.results(), _run(dm, wl, flags=sl.FLAG_ROW_KERNELS | sl.FLAG_UNGROUPED_ROWS))
    dm.free()


@pytest.mark.parametrize("dtype,n,last", [
    ("bf16", 203, 512), ("bf16", 204, 512),   # lists of 307 entries: 1624 and 1632 blocks of 64 nodes, shared below 1628
    ("f32", 203, 508), ("f32", 204, 508),
    ("bf16", 148, 505), ("bf16", 147, 505),   # a load of one node: shared below 1184 blocks
])
def test_plain_layers_share_a_walk_by_the_length_of_their_lists(dtype, n, last):
    """One block per (query, 64 nodes) or per query, at budgets that always go by input."""
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(5100 + n, [64, 2048, last], [1, 0], dtype, n=n, n_cal=200, K=4, L=2, budgets=(20, 700, 1500))
    dm = harness.DeviceModel(wl)
    _same_bits(_run(dm, wl), _run(dm, wl, flags=sl.FLAG_ROW_KERNELS | sl.FLAG_UNGROUPED_ROWS))
    dm.free()


def test_grouped_products_need_their_scratch_and_do_without_it():
    """A workspace of the size the other kernels need is still taken, with the same results."""
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(4202, [128, 512, 256, 20], [1, 1, 0], "f32", n=600, n_cal=300, K=4, L=2, budgets=(2500, 6000))
    dm = harness.DeviceModel(wl)
    small = sl.slonn_workspace_bytes(dm.model, 600, 6000, flags=sl.FLAG_ROW_KERNELS)
    assert small < sl.slonn_workspace_bytes(dm.model, 600, 6000)
    _same_bits(_run(dm, wl), _run(dm, wl, ws_bytes=small))
    dm.free()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_grouped_products_keep_queries_apart(dtype):
    """Infinities and NaNs in some queries stay in those queries; the others, in the same groups, are untouched."""
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(4203, [128, 256, 264, 40], [1, 1, 0], dtype, n=320, n_cal=300, K=2, L=2, budgets=(6000,))
    dm = harness.DeviceModel(wl)
    clean = _run(dm, wl)
    x = wl.x.copy()
    x[5::7, 3] = np.inf
    x[6::7, 9] = np.nan
    dirty = _run(dm, wl, x=x)
    rows = _run(dm, wl, flags=sl.FLAG_ROW_KERNELS, x=x)
    for k in KEYS:
        assert np.array_equal(dirty[k], rows[k], equal_nan=dirty[k].dtype == np.float32), k
    others = [q for q in range(320) if q % 7 not in (5, 6)]
    assert np.array_equal(clean["logits"][others], dirty["logits"][others])
    dm.free()


@pytest.mark.parametrize("dims,has_act,n,budgets,max_bp", [
    ([512, 640, 520, 24], [1, 1, 0], 600, (1500, 2500, 6000), 6000),    # grouped rows, grouped products, plain last layer
    ([512, 640, 520, 300], [1, 1, 1], 600, (2500, 6000), 6000),         # budgeted last layer
    ([512, 640, 520, 24], [1, 1, 0], 600, (1500, 3000), 3000),          # both budget classes of the compacted row groups in one
    ([512, 640, 520, 24], [1, 1, 0], 600, (2500, 6000, 10000), 10000),  # beside 100 % queries on their own route
    ([512, 640, 520, 24], [1, 1, 0], 2100, (600, 800, 2500), 2500),     # groups sorted from a low budget on
])
def test_budgets_above_the_maximum_get_the_clamped_results(dims, has_act, n, budgets, max_bp):
    """A query whose budget is too large is reported and evaluated at the batch's maximum, whatever kernels the batch takes; the
    output buffers hold something else before the run."""
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(4500 + n, dims, has_act, "bf16", n=n, n_cal=300, K=4, L=2, budgets=budgets)
    dm = harness.DeviceModel(wl)
    bad = {7: 20000, 8: 65535, 70: 10001, 71: 0, n - 1: max_bp + 1}
    bp, clamped = wl.budget_bp.copy(), wl.budget_bp.copy()
    for q, v in bad.items():
        bp[q], clamped[q] = v, 1 if v == 0 else max_bp
    want = harness.run_once(dm, wl.x, clamped, max_budget_bp=max_bp, kernel_path=1, flags=sl.FLAG_ROW_KERNELS | sl.FLAG_UNGROUPED_ROWS)
    for flags in (0, sl.FLAG_ROW_KERNELS, sl.FLAG_ROW_KERNELS | sl.FLAG_UNGROUPED_ROWS):
        b = harness.DeviceBatch(dm, wl.x, bp, max_budget_bp=max_bp, kernel_path=1, flags=flags)
        b.logits.fill_(777.0)
        b.vals.fill_(777.0)
        b.pred.fill_(7777)
        b.run()
        got = b.results()
        assert got["status"][0] == 5 and got["status"][1] in bad
        ip = want["active_indptr"].astype(np.int64)
        assert np.array_equal(got["active_indptr"], want["active_indptr"])
        for k in ("pred", "codes", "active_ids", "active_vals"):
            assert np.array_equal(got[k], want[k]), (flags, k)
        for q in range(n):
            B = int(ip[(q + 1) * sum(has_act)] - ip[(q + 1) * sum(has_act) - 1]) if has_act[-1] else dims[-1]
            assert np.array_equal(got["logits"][q, :B], want["logits"][q, :B]), (flags, q)
    dm.free()


def test_launch_records_say_which_launches_took_grouped_products():
    """What the benchmark names and counts kernels by: launches that read single weights of a transposed copy carry
    cols_bp = 10000, the row kernels 0."""
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    wl = custom_workload(4204, [512, 1240, 520, 120], [1, 1, 0], "bf16", n=3500, n_cal=300, K=4, L=2, budgets=(700, 5000, 10000))
    dm = harness.DeviceModel(wl)
    sh = acc.NetShape.of(wl)

    def kernels(flags):
        b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED, flags=flags)
        recs = sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes)
        assert b.results()["status"][0] == 0
        return {(r["layer"], acc.kernel_name(sh, r), r["bp_lo"] == 10000) for r in recs if r["layer"] is not None}

    tiled, rows = kernels(0), kernels(sl.FLAG_ROW_KERNELS)
    assert {(0, "tile_rows_kernel", True), (1, "tile_rows_kernel", True), (2, "tile_rows_kernel", True),
            (1, "hash_select_cols_kernel", False), (1, "tile_rows_kernel", False), (2, "tile_rows_kernel", False)} <= tiled
    assert not [k for k in rows if k[1] in ("tile_rows_kernel", "hash_select_cols_kernel")]
    dm.free()


@pytest.mark.parametrize("dtype,dims,has_act,n,budgets,K,L", [
    ("bf16", [4096, 2048, 24], [1, 0], 8192 + 40, (1500, 1876, 1900), 4, 2),        # groups of four sorted below 20 %, two chunks
    ("bf16", [512, 640, 520, 24], [1, 1, 0], 8192 + 309, (600, 2001, 2500), 4, 2),  # from 20 % on
    ("f32", [264, 512, 512, 20], [1, 1, 1], 8192 + 33, (700, 2500, 10000), 4, 2),   # 100 % queries beside them
    ("bf16", [128, 640, 520, 20], [1, 1, 0], 300, (2500, 6000), 9, 4),              # 36 hash functions: no side-by-side hash rows
    ("f32", [128, 640, 520, 44], [1, 1, 1], 2100, (700, 6000), 9, 4),
])
def test_sorted_groups_and_many_hash_functions(dtype, dims, has_act, n, budgets, K, L):
    """Against the row kernels, which neither sort nor read by input."""
    from paper_2204_08400_b200 import binding as sl, harness
    wl = custom_workload(4700 + n, dims, has_act, dtype, n=n, n_cal=600, K=K, L=L, budgets=budgets)
    dm = harness.DeviceModel(wl)
    _same_bits(_run(dm, wl), _run(dm, wl, flags=sl.FLAG_ROW_KERNELS | sl.FLAG_UNGROUPED_ROWS))
    dm.free()


@pytest.mark.parametrize("dtype,dims,has_act,n,budgets,layer,kernel", [
    ("bf16", [512, 640, 640, 10], [1, 1, 0], 2100, (1000, 5000), 2, None),              # a tile of 128 columns for 10 nodes
    ("bf16", [512, 640, 640, 95], [1, 1, 0], 2100, (1000, 5000), 2, None),
    ("bf16", [512, 640, 640, 96], [1, 1, 0], 2100, (1000, 5000), 2, "tile_rows_kernel"),
    ("bf16", [512, 640, 640, 96], [1, 1, 0], 1500, (1000, 5000), 2, None),              # 94 items
    ("bf16", [512, 640, 640, 256], [1, 1, 0], 2100, (500, 1999), 2, None),              # low budgets behind the second layer ...
    ("bf16", [512, 640, 640, 256], [1, 1, 0], 2100, (500, 2000), 2, "tile_rows_kernel"),
    ("bf16", [512, 640, 640, 640, 256], [1, 1, 1, 0], 2100, (500, 1999), 3, "tile_rows_kernel"),   # ... and behind the third
    ("f32", [128, 2048, 256], [1, 0], 1000, (500, 1000), 1, "tile_rows_kernel"),        # wide and fp32
    ("f32", [128, 2040, 256], [1, 0], 1000, (500, 1000), 1, None),
    ("bf16", [512, 1536, 24], [1, 0], 2100, (1900,), 0, "gather_dot_kernel"),           # 0.3 MB of selected rows a query
    ("bf16", [4096, 2048, 24], [1, 0], 2100, (1875, 1876), 0, "group_rows_kernel"),     # 3 MiB from 18.75 % on
    ("bf16", [512, 1536, 1536, 24], [1, 1, 0], 2100, (2900,), 1, "layer_cols_kernel"),  # 445 nodes in the first list-fed layer,
    ("bf16", [512, 1536, 1536, 1536, 1536, 24], [1, 1, 1, 1, 0], 2100, (2900,), 3, "tile_rows_kernel"),  # in the third,
    ("bf16", [512, 1536, 1536, 24], [1, 1, 0], 2100, (2900, 5000), 1, "tile_rows_kernel"),  # and beside higher budgets
])
def test_grouped_products_are_taken_where_they_pay(dtype, dims, has_act, n, budgets, layer, kernel):
    """Both sides of each line of the dispatch (None: anything but grouped products); same bits as the row kernels."""
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    wl = custom_workload(4800 + n, dims, has_act, dtype, n=n, n_cal=300, K=4, L=2, budgets=budgets)
    dm = harness.DeviceModel(wl)
    b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED)
    names = [acc.kernel_name(acc.NetShape.of(wl), r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes)
             if r["layer"] == layer and r["bp_lo"] <= budgets[0 if len(budgets) > 1 and budgets[0] == 2900 else -1] <= r["bp_hi"]]
    if kernel:
        assert names[-1] == kernel, names
    else:
        assert "tile_rows_kernel" not in names, names
    _same_bits(b.results(), _run(dm, wl, flags=sl.FLAG_ROW_KERNELS | sl.FLAG_UNGROUPED_ROWS))
    dm.free()


@pytest.mark.parametrize("dtype,dims,has_act,n,budgets,layer,kernel", [
    ("bf16", [640, 96, 24], [0, 1], 2100, (1000, 5000), 0, "tile_rows_kernel"),
    ("bf16", [640, 256, 24], [0, 1], 2100, (1000, 5000), 0, "tile_rows_wide_kernel"),      # every node, eight columns per load
    ("f32", [640, 256, 24], [0, 1], 2100, (1000, 5000), 0, "tile_rows_wide_kernel"),
    ("f32", [640, 252, 24], [0, 1], 2100, (1000, 5000), 0, "tile_rows_kernel"),            # a load of four columns, but not of eight
    ("f32", [40, 1000, 24], [0, 1], 3000, (1000, 5000), 0, "tile_rows_wide_kernel"),       # four items a group, the last not full; stretches without inputs
    ("bf16", [2512, 2080, 24], [0, 1], 1150, (5000,), 0, "tile_rows_wide_kernel"),         # 5 and 9 rounds of items, 9.97 MiB
    ("bf16", [2560, 2080, 24], [0, 1], 1150, (5000,), 0, "tile_rows_kernel"),              # 10.2 MiB
    ("f32", [2512, 1040, 24], [0, 1], 880, (5000,), 0, "tile_rows_wide_kernel"),           # 2 and 4
    ("f32", [2560, 1040, 24], [0, 1], 880, (5000,), 0, "tile_rows_kernel"),
    ("f32", [2560, 1040, 24], [0, 1], 1408, (5000,), 0, "tile_rows_wide_kernel"),          # 3 and 6
    ("f32", [2560, 4104, 24], [0, 1], 1408, (5000,), 0, "tile_rows_kernel"),               # 40.1 MiB
    ("bf16", [64, 512, 504], [1, 0], 8192, (1000, 5000), 1, "tile_rows_wide_kernel"),      # behind lists: 7 rounds,
    ("bf16", [64, 512, 504], [1, 0], 7000, (1000, 5000), 1, "tile_rows_kernel"),           # 6
])
def test_which_product_kernel_is_taken(dtype, dims, has_act, n, budgets, layer, kernel):
    """The launch records tell the kernels with 128 and 256 columns per work item apart; same bits as the row kernels."""
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    wl = custom_workload(4900 + n, dims, has_act, dtype, n=n, n_cal=300, K=4, L=2, budgets=budgets)
    dm = harness.DeviceModel(wl)
    b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED)
    names = [acc.timed_kernel(acc.NetShape.of(wl), r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes) if r["layer"] == layer]
    assert names[-1] == kernel, names
    _same_bits(b.results(), _run(dm, wl, flags=sl.FLAG_ROW_KERNELS | sl.FLAG_UNGROUPED_ROWS))
    dm.free()


@pytest.mark.parametrize("dtype,dims,has_act,n,budgets,layer,lo,kernel", [
    ("bf16", [512, 1240, 520, 120], [1, 1, 0], 3500, (10000,), 0, 10000, "tile_rows_wide_kernel"),  # ids written, a last load clamped
    ("f32", [512, 1240, 520, 120], [1, 1, 0], 3500, (10000,), 0, 10000, "tile_rows_wide_kernel"),
    ("bf16", [512, 1240, 512, 120], [1, 1, 0], 3500, (10000,), 1, 10000, "tile_rows_wide_kernel"),           # complete lists
    ("bf16", [512, 1240, 505], [1, 0], 3500, (10000,), 1, 10000, "tile_rows_kernel"),                        # one column per load
    ("bf16", [512, 1240, 520, 120], [1, 1, 0], 3500, (700, 10000), 0, 10000, "tile_rows_wide_kernel"),       # about half of the groups
    ("bf16", [512, 1240, 520, 120], [1, 1, 0], 3500, (700,) * 19 + (10000,), 0, 10000, "tile_rows_kernel"),  # a dozen groups of 219
    # selected nodes: 2304 items and (a second chunk, of few groups) 1950; one column more than four items hold
    ("bf16", [64, 520, 1032, 24], [1, 1, 0], 8192, (9000, 9999), 1, 3501, "tile_rows_wide_kernel"),
    ("f32", [64, 516, 1032, 24], [1, 1, 0], 8192 + 800, (9000, 9999), 1, 3501, "tile_rows_wide_kernel"),
    ("bf16", [64, 72, 1028], [1, 1], 8192, (9000, 9999), 1, 3501, "tile_rows_wide_kernel"),   # partial sums without an input
    ("bf16", [64, 520, 1032, 24], [1, 1, 0], 8192, (500,) * 15 + (9999,), 1, 3501, "tile_rows_kernel"),
    ("bf16", [64, 520, 1032, 24], [1, 1, 0], 7000, (9000,), 1, 3501, "tile_rows_kernel"),            # 1752
])
def test_item_width_follows_the_queries_that_are_served(dtype, dims, has_act, n, budgets, layer, lo, kernel):
    """A few queries of a large batch leave few work items: the kernel whose items are shorter; same bits as the row kernels."""
    from paper_2204_08400_b200 import accounting as acc, binding as sl, harness
    wl = custom_workload(5000 + n, dims, has_act, dtype, n=n, n_cal=300, K=4, L=2, budgets=budgets)
    dm = harness.DeviceModel(wl)
    b = harness.DeviceBatch(dm, wl.x, wl.budget_bp, kernel_path=sl.PATH_STAGED)
    sh = acc.NetShape.of(wl)
    names = [acc.timed_kernel(sh, r) for r in sl.slonn_run_traced(dm.model, b.batch, b.ws, b.ws_bytes)
             if r["layer"] == layer and r["bp_lo"] == lo and acc.grouped_products(r)]
    assert names == [kernel], names
    _same_bits(b.results(), _run(dm, wl, flags=sl.FLAG_ROW_KERNELS | sl.FLAG_UNGROUPED_ROWS))
    dm.free()
