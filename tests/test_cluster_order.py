"""Distributed shared memory: a CTA may write another CTA's shared memory only
after a barrier of the cluster has shown that that CTA has started, and no CTA may
leave while another one can still write its memory. No run can show a missing
barrier (it works by latency), so the order is read from the kernel's source."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _kernel_body():
    text = open(os.path.join(ROOT, "paper_2401_04068_gb300", "csrc", "resident.cu")).read()
    text = re.sub(r"//[^\n]*", "", text)
    start = text.index("{", text.index("bellman_cluster_kernel(StepLaunch"))
    depth = 0
    for i in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[start:i + 1]
    raise AssertionError("unbalanced braces")


def test_cluster_barrier_before_the_first_remote_store():
    body = _kernel_body()
    first_store = body.index("st_remote(")
    assert "cluster_sync(size);" in body[:body.index("for (int j = 0;;")]
    assert body.index("cluster_sync(size);") < first_store


def test_no_remote_store_between_the_last_barrier_and_the_exit():
    # the loop is left right behind the barrier that follows rank 0's store of the next unit
    body = _kernel_body()
    leave = body.index("if (u >= R.n_units) break;")
    assert body.rindex("cluster_sync(size);", 0, leave) > body.rindex("st_remote(", 0, leave)
    assert "st_remote(" not in body[body.index("S.is_last"):]
