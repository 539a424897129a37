"""A cluster of 16 blocks may be too large for a device that is shared.  The form whose list-fed layers run input-stationary needs more
shared memory than the one that reads whole rows, so the latter is tried where the former cannot be scheduled.  Checked on the
sources: on a device of its own both fit."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2204_08400_b200", "csrc")


def test_the_row_form_is_tried_where_the_other_cannot_be_scheduled():
    with open(os.path.join(CSRC, "slonn_run.cu")) as f:
        run = re.sub(r"//[^\n]*", "", f.read())
    body = run[run.index("int launch_cluster(const slonn_model"):]
    body = body[:body.index("\n}\n")]
    first = body.index("cluster_lists_kernel<true>")
    second = body.index("cluster_network_kernel<true, SLONN_CLUSTER_THREADS")
    assert first < second
    between = body[body.rindex(";", 0, first) + 1:second]
    assert re.search(r"const int rc = launch_cluster_t\(", between), "its result is looked at"
    assert "if (rc != SLONN_ERR_DIM) return rc;" in between
    assert re.findall(r"return [^;]*;", between) == ["return rc;"], "and nothing else leaves in between"
