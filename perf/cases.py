"""The work a user of this library has it do, as timed cases.

A case is one pass through a public entry point (`slonn_run` for a batch that is on the device, `slonn_run_host` for
one in host memory, `slonn_build` + `slonn_serialize` for training an activator), on a network of the shapes the
benchmark and the tests use.  Weights, calibration rows and queries are drawn on the device from the seed.

A case is a dict of
    net, act        layer widths "D0-N1-...-Nout"; per layer "1" = carries a Node Activator
    dtype           storage type of the weights, "bf16" or "f32"
    law             "half_zero": uniform [0, 1) with half of the values exactly 0 (image-like rows);
                    "relu_normal": max(N(0, 1), 0); "csr75": CSR rows of 75 nonzeros, log-normal values
    queries, calib  rows of the batch, and rows the activator is trained on
    budgets         basis points, one value for the whole batch or several drawn per query ("500,1000,2500")
    lists           1: the caller wants hash codes and active lists back, 0: logits and predictions only
    call            "run", "host" or "build"
    dense_tc        1: queries at 10000 bp run on the tensor cores (SLONN_FLAG_DENSE_TC)
    free_hash       1: hash nodes always active and absent from the lists
    list_cap        entries kept per bucket list, 0 = all
"""
import math

import torch

from paper_2204_08400_b200 import binding as sl

DEVICE = "cuda:0"
K, L = 10, 2                                   # key bits and tables: the paper's default
DEEP = "4096-4096-4096-4096-4096-4096-4096-4096-4096-1000"
DEEP_ACT = "111111110"
MIXED = "500,1000,2500,5000,10000"


def _case(net, act, dtype, law, queries, calib, budgets, lists=0, call="run", dense_tc=0, free_hash=0, list_cap=0, name=None):
    c = dict(net=net, act=act, dtype=dtype, law=law, queries=queries, calib=calib, budgets=budgets, lists=lists, call=call,
             dense_tc=dense_tc, free_hash=free_hash, list_cap=list_cap)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # an interactive request on a deep network: one query, answered as soon as possible
        _case(DEEP, DEEP_ACT, "bf16", "relu_normal", 1, 1024, "1000", name="deep_1q_10pct"),
        # a small server batch on the same network at a middle budget
        _case(DEEP, DEEP_ACT, "bf16", "relu_normal", 64, 1024, "2500", name="deep_64q_25pct"),
        # throughput serving of the deep network at a low budget: the benchmark's headline batch
        _case(DEEP, DEEP_ACT, "bf16", "relu_normal", 4096, 1024, "1000", name="deep_4096q_10pct"),
        # the same batch where accuracy matters more: half of the nodes
        _case(DEEP, DEEP_ACT, "bf16", "relu_normal", 4096, 1024, "5000", name="deep_4096q_50pct"),
        # the headline batch as a service sees it: queries and results in pinned host memory
        _case(DEEP, DEEP_ACT, "bf16", "relu_normal", 4096, 1024, "1000", call="host", name="deep_4096q_10pct_host"),
        # a stream of requests with service levels of their own, from 5 % to the full network
        _case("2048-4096-4096-1000", "110", "bf16", "relu_normal", 8192, 2048, MIXED, name="mixed_slo_8192q"),
        # the full network for every query, on the tensor cores: the baseline a user compares against
        _case("2048-4096-4096-1000", "110", "bf16", "relu_normal", 8192, 2048, "10000", dense_tc=1, name="full_tc_8192q"),
        # offline scoring of a data set with a narrow network
        _case("784-1024-1024-10", "110", "bf16", "half_zero", 65536, 4096, "1000", name="narrow_65536q_10pct"),
        # the paper's image classifier, fp32, a thousand queries, with the active lists handed back
        _case("784-112-112-10", "110", "f32", "half_zero", 1024, 4096, "2500", lists=1, name="image_1024q_25pct_lists"),
        # extreme classification: sparse text-like rows, 200,000 budgeted outputs
        _case("100000-128-200000", "01", "f32", "csr75", 256, 2048, "500", name="extreme_256q_5pct"),
        # widths that are no powers of two, an odd batch, every layer budgeted (the output too), lists handed back
        _case("2328-1568-1656-595", "111", "bf16", "relu_normal", 777, 1024, "700,1500,3000,6000", lists=1, name="ragged_777q_lists"),
        # training a node activator (Algorithm 1) and saving it
        _case("784-1024-1024-10", "110", "bf16", "half_zero", 1, 16384, "1000", call="build", name="build_narrow_16384rows"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _width(rng, lo, hi, mult=8):
    return max(mult, int(round(_log(rng, lo, hi) / mult)) * mult)


def draw(rng):
    kind = rng.choice(["wide", "wide", "wide", "narrow", "narrow", "extreme"])
    lists = int(rng.random() < 0.3)
    free_hash = int(rng.random() < 0.15)
    dtype = "bf16" if rng.random() < 0.7 else "f32"
    one = [500, 1000, 1500, 2500, 3500, 5000, 10000]
    mixed = [MIXED, "700,1500,3000,6000", "1000,2500"]
    if kind == "extreme":
        return _case("%d-%d-%d" % (_width(rng, 20000, 100000), _width(rng, 64, 256), int(_log(rng, 20000, 200000))), "01", "f32", "csr75",
                     int(_log(rng, 16, 256)), int(rng.randint(256, 2048)), str(rng.choice([100, 500, 1000])), lists=lists)
    budgets = rng.choice(mixed) if rng.random() < 0.4 else str(rng.choice(one))
    if kind == "narrow":
        w1, w2 = _width(rng, 96, 1024), _width(rng, 96, 1024)
        dims = [rng.choice([784, _width(rng, 256, 1024)]), w1, w2, rng.randint(10, 100)]
        act, law, queries = "110", "half_zero", int(_log(rng, 256, 65536))
    else:
        depth = rng.randint(2, 8)
        width = _width(rng, 512, 4096)
        ragged = rng.random() < 0.3
        dims = [_width(rng, 512, 4096)] + [_width(rng, 512, 4096) if ragged else width for _ in range(depth)] + [rng.randint(100, 1000)]
        act, law, queries = "1" * depth + rng.choice("001"), "relu_normal", int(_log(rng, 1, 8192))
    # no larger than the largest listed case: whole rows of the selected nodes, in multiply-adds
    top = max(int(b) for b in budgets.split(","))
    per_query = sum(dims[l] * dims[l + 1] * (top if act[l] == "1" else 10000) / 10000 for l in range(len(act)))
    queries = max(1, min(queries, int(1.2e11 / per_query)))
    call = "host" if rng.random() < 0.15 and not lists else "run"
    dense_tc = int(top == 10000 and dtype == "bf16" and act[-1] == "0" and call == "run" and not lists and rng.random() < 0.3)
    return _case("-".join(str(d) for d in dims), act, dtype, law, queries, rng.randint(256, 2048), budgets, lists=lists, call=call,
                 dense_tc=dense_tc, free_hash=0 if dense_tc else free_hash)


# ---- inputs ---------------------------------------------------------------------------

def _dense_rows(n, d, law, g):
    if law == "half_zero":
        x = torch.rand((n, d), generator=g, device=DEVICE)
        return torch.where(torch.rand((n, d), generator=g, device=DEVICE) < 0.5, x, torch.zeros((), device=DEVICE))
    return torch.randn((n, d), generator=g, device=DEVICE).clamp_(min=0)


def _csr_rows(n, d, nnz, g):
    """nnz distinct ascending ids per row: one from each of nnz equal stretches of the columns."""
    step = d // nnz
    ids = torch.arange(nnz, device=DEVICE) * step + torch.randint(0, step, (n, nnz), generator=g, device=DEVICE)
    vals = torch.randn((n, nnz), generator=g, device=DEVICE).exp_()
    indptr = torch.arange(n + 1, dtype=torch.int64, device=DEVICE) * nnz
    return indptr, ids.to(torch.int32).reshape(-1).contiguous(), vals.reshape(-1).contiguous()


class _State:
    """What a serving program keeps: weights, the built model, the batch's buffers."""


def prepare(case, seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(seed)
    s = _State()
    s.case = dict(case)
    dims = [int(d) for d in case["net"].split("-")]
    act = [int(a) for a in case["act"]]
    n, csr = case["queries"], case["law"] == "csr75"
    s.dims, s.act = dims, act
    s.dtype = sl.SLONN_BF16 if case["dtype"] == "bf16" else sl.SLONN_F32
    s.W, s.bias = [], []
    for d, m in zip(dims[:-1], dims[1:]):
        w = torch.randn((m, d), generator=g, device=DEVICE).mul_(math.sqrt(2.0 / d))
        s.W.append(w.to(torch.bfloat16) if case["dtype"] == "bf16" else w)
        s.bias.append(torch.zeros(m, device=DEVICE))
    s.build_args = dict(K=K, L=L, list_cap=case["list_cap"], seed=seed, first_layer_sparse=csr, free_hash_nodes=bool(case["free_hash"]))
    rows = _csr_rows(case["calib"], dims[0], 75, g) if csr else _dense_rows(case["calib"], dims[0], case["law"], g)
    s.build_args["calib_csr" if csr else "calib_dense"] = rows
    if case["call"] == "build":
        torch.cuda.synchronize()
        return s
    torch.cuda.synchronize()
    s.model = sl.slonn_build(dims, act, s.dtype, s.W, s.bias, **s.build_args)
    s.build_args = None

    choices = [int(b) for b in case["budgets"].split(",")]
    top = max(choices)
    pick = torch.randint(0, len(choices), (n,), generator=g, device=DEVICE)
    bp = torch.tensor(choices, dtype=torch.int16, device=DEVICE)[pick]
    x = None if csr else _dense_rows(n, dims[0], case["law"], g)
    s.x_csr = _csr_rows(n, dims[0], 75, g) if csr else None
    stride = sl.slonn_logit_stride(s.model, top)
    host = case["call"] == "host"

    def buffer(shape, dtype):
        t = torch.zeros(shape, dtype=dtype, device="cpu" if host else DEVICE)
        return t.pin_memory() if host else t

    s.x = x.cpu().pin_memory() if host else x
    s.bp = bp.cpu().pin_memory() if host else bp
    s.out = dict(logits=buffer((n, stride), torch.float32), pred=buffer((n,), torch.int32), status=buffer((4,), torch.int32))
    extra = {}
    if act[-1]:
        s.out["logit_ids"] = buffer((n, stride), torch.int32)
        extra["logit_ids"] = s.out["logit_ids"]
    if case["lists"]:
        cap = sl.slonn_active_capacity(s.model, n, top)
        s.out["codes"] = buffer((n, sum(act), L), torch.int16)
        s.out["active_indptr"] = buffer((n * sum(act) + 1,), torch.int64)
        s.out["active_ids"] = buffer((cap,), torch.int32)
        s.out["active_vals"] = buffer((cap,), torch.float32)
        for k in ("codes", "active_indptr", "active_ids", "active_vals"):
            extra[k] = s.out[k]
    flags = sl.FLAG_DENSE_TC if case["dense_tc"] else 0
    s.batch = sl.make_batch(n, s.bp, s.out["logits"], s.out["status"], x_dense=s.x, x_csr=s.x_csr, max_budget_bp=top,
                            pred=s.out["pred"], flags=flags, **extra)
    size = sl.slonn_host_workspace_bytes if host else sl.slonn_workspace_bytes
    s.ws_bytes = size(s.model, n, top, flags=flags)
    s.ws = torch.empty(s.ws_bytes, dtype=torch.uint8, device=DEVICE)
    return s


def run(s):
    stream = torch.cuda.current_stream().cuda_stream
    call = s.case["call"]
    if call == "build":
        model = sl.slonn_build(s.dims, s.act, s.dtype, s.W, s.bias, stream=stream, **s.build_args)
        blob = sl.slonn_serialize(model)
        sl.slonn_free(model)
        return {"activator": blob}
    if call == "host":
        sl.slonn_run_host(s.model, s.batch, s.ws, s.ws_bytes, stream)
    else:
        sl.slonn_run(s.model, s.batch, s.ws, s.ws_bytes, stream)
    return s.out


# ---- what a pass cannot do without ----------------------------------------------------

def _nodes(bp, width):
    return min(width, max(1, (bp * width + 5000) // 10000))


def work(case):
    """Bytes: the queries in, the results out, the weight rows that at least one query selects (at most all of them) and
    their bucket lists, each once.  Operations: two per selected node and input the layer below handed over."""
    dims = [int(d) for d in case["net"].split("-")]
    act = [int(a) for a in case["act"]]
    esz = 2 if case["dtype"] == "bf16" else 4
    n = case["calib"] if case["call"] == "build" else case["queries"]
    choices = [10000] if case["call"] == "build" else [int(b) for b in case["budgets"].split(",")]
    csr = case["law"] == "csr75"
    total_bytes = n * (75 * 8 if csr else dims[0] * 4)
    flops = 0.0
    for l in range(len(act)):
        d, m = dims[l], dims[l + 1]
        out = [_nodes(b, m) if act[l] else m for b in choices]
        fed = [75 if csr and l == 0 else _nodes(b, d) if l and act[l - 1] else d for b in choices]
        flops += 2.0 * n * sum(o * f for o, f in zip(out, fed)) / len(choices)
        total_bytes += min(m, n * max(out)) * min(d, n * max(fed)) * esz
        if act[l]:
            ids = 2 if m <= 65536 else 4
            flops += 2.0 * n * K * L * sum(fed) / len(choices)
            total_bytes += L * max(out) * ids * min(n, 1 << K)
            if case["lists"]:
                total_bytes += n * (sum(out) / len(choices) * 8 + L * 2)
    if case["call"] != "build":
        total_bytes += n * (dims[-1] if not act[-1] else _nodes(max(choices), dims[-1])) * 4 + n * 4
    return {"bytes": int(total_bytes), "flops": flops}


def tolerance(case):
    """The order of every sum is part of the interface (32 partial sums, fixed tree), so results are the same bits
    whatever kernel forms them.  Only the tensor-core route leaves the order open: activations are rounded to bf16
    between layers there, and another order of the fp32 sums moves some of them to the neighbouring value.  Measured
    against the same network with fp64 sums (three seeds): 4.1e-4 of the norm, 5.8e-3 of the root mean square at most,
    0.13 % of the predictions (near ties); stated are about four times these."""
    if case["dense_tc"]:
        return {"rel": 1.6e-3, "max": 2.4e-2, "differ": 6e-3}
    return "exact"
