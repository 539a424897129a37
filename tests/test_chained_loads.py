"""A run's kernels are chained: one may be resident while the kernel before it still writes.  What kernels of the chain write
must therefore be read with plain loads (ordered by the wait they begin with), never through the read-only path, which is for
memory nobody writes while a kernel is resident.  Checked on the sources: the order of the two is up to the hardware and a
wrong one need not show."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2204_08400_b200", "csrc")
FILES = sorted(os.path.basename(p) for p in glob.glob(os.path.join(CSRC, "*.cuh"))) + ["slonn_run.cu", "slonn_dense_tc.cu"]
# members and arguments that hold what a kernel of the chain wrote
WRITTEN = {"dense", "ids", "vals", "indptr", "idlist", "order", "list", "count", "work", "items", "kseg", "krow", "xt", "ucol",
           "ucount", "bm", "pre", "key", "sort_key", "ent", "seg", "gseg", "nodes", "quads", "out_ids", "out_vals", "tile_sums", "logits", "row_count", "row_map"}


def read_only_loads(text):
    """(argument, names in it, local pointers set from what the chain writes) of every __ldg in the text."""
    text = re.sub(r"//[^\n]*", "", text)
    for body in re.split(r"(?=\b__global__\b|\b__device__\b)", text):
        aliases = {m.group(1) for m in re.finditer(r"\*\s*(?:const\s+)?(\w+)\s*=\s*([^;]*);", body)
                   if WRITTEN & set(re.findall(r"\w+", re.sub(r"\w+\[[^\]]*\]", "", m.group(2))))}
        for m in re.finditer(r"__ldg\(", body):
            depth, end = 1, m.end()
            while depth:
                depth += {"(": 1, ")": -1}.get(body[end], 0)
                end += 1
            arg = body[m.end():end - 1]
            base = re.sub(r"\[[^\]]*\]|\b\w+\s*\(", "", arg)          # an index, a cast or a call is not what is loaded from
            yield arg, set(re.findall(r"\w+", base.split("+")[0])), aliases


@pytest.mark.parametrize("name", FILES)
def test_what_the_chain_writes_is_read_with_plain_loads(name):
    with open(os.path.join(CSRC, name)) as f:
        loads = list(read_only_loads(f.read()))
    bad = [arg for arg, names, aliases in loads if names & (WRITTEN | aliases)]
    assert not bad, bad


def test_the_check_sees_direct_and_renamed_loads():
    for body in ("__device__ void f() { const float4 *src = (const float4 *)(in.dense + q); v = __ldg(src + i); }",
                 "__global__ void k(P p) { x = __ldg(P.ids + off + r); }",
                 "__global__ void k(P p) { const uint2 *at = Q.quads + q * Q.quad_stride; v = __ldg(at + r0); }",
                 "__global__ void k(P p) { seg[tid] = __ldg(gseg + tid); v = __ldg(Q.ent + i); }",
                 "__global__ void k(P p) { const float *vals = P.in.vals + s; x = in ? __ldg(vals + i) : 0.0f; }"):
        arg, names, aliases = next(iter(read_only_loads(body)))
        assert names & (WRITTEN | aliases), body
    arg, names, aliases = next(iter(read_only_loads("__global__ void k(P p) { b = __ldg(P.bias + P.ids[r]); }")))
    assert not names & (WRITTEN | aliases)


def test_a_chain_starts_behind_a_full_dependency():
    """What a caller's own kernel may just be writing is read through the read-only path only behind a memset of the call's own; an
    entry point without one does not chain its kernel."""
    with open(os.path.join(CSRC, "slonn_run.cu")) as f:
        run = f.read()
    body = run[run.index("static int run_impl("):]
    assert body.index("cudaMemsetAsync(b->status") < body.index("slonn_launch(")
    assert body.index("cudaMemsetAsync(b->status") < body.index("launch_cluster(")
    with open(os.path.join(CSRC, "slonn_dense_tc.cu")) as f:
        tc = f.read()
    entry = tc[tc.index('extern "C" int slonn_dense_layer('):]
    assert "(cudaStream_t)stream, false);" in entry, "slonn_dense_layer works without a status buffer, hence without a memset"


def test_no_kernel_lets_the_next_one_in_early():
    """Blocks of the next kernel would wait in slots that another stream's blocks could use."""
    for name in FILES:
        with open(os.path.join(CSRC, name)) as f:
            code = re.sub(r"//[^\n]*", "", f.read())
        assert "launch_dependents" not in code and "TriggerProgrammaticLaunch" not in code, name
