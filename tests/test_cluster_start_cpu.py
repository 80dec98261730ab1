"""Distributed shared memory may be written only once the block that owns it has started. The blocks of a
cluster solve write their partial sums to each other, so the solver's kernel has to meet its cluster's barrier
before the first of those stores, and the barrier's aligned form wants whole warps. Whether a block was late
shows in no result, so the order is read from the source."""

import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2204_14241_gb300", "csrc")


def code(name):
    with open(os.path.join(SRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def body(text, head):
    """The braces that follow the first match of `head`."""
    i = text.index("{", re.search(head, text).end())
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j + 1]
    raise AssertionError("unbalanced braces")


def test_cluster_barrier_before_the_first_remote_store():
    text = code("team.cu")
    assert "barrier.cluster.arrive.release" in body(text, r"void cluster_sync\(\)")
    kernel = body(text, r"\bk_team\(")
    first = re.search(r"if constexpr \(CLU\) cluster_sync\(\);", kernel)
    assert first and first.start() < kernel.index("team_run<")
    for helper in ("pre_tables<", "sync_sum<"):
        if helper in kernel:
            assert first.start() < kernel.index(helper)


def test_whole_warps_at_the_cluster_barrier():
    reduction = body(code("team.cu"), r"\bsync_sum\(")
    store = reduction.index("st.shared::cluster")
    assert "__syncwarp();" in reduction[store:reduction.index("cluster_sync();", store)]
