"""Orderings between threads that no run can show to be missing (the hardware mostly supplies them by
itself), read off the CUDA sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2406_01911_gb300", "csrc")


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def body(text, head):
    """The braces' contents that follow `head`."""
    i = text.index("{", text.index(head))
    depth = 0
    for j in range(i, len(text)):
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        if depth == 0:
            return text[i:j]
    raise AssertionError(head)


def test_cluster_meets_before_the_first_remote_store():
    """A block may write into another block's shared memory only once that block runs."""
    k = body(source("greedy.cu"), "k_greedy(GreedyParams P)")
    assert k.index("grid_meet<kCluster>") < k.index("send_winner")


def test_cluster_barrier_takes_a_diverged_warp():
    """.aligned asks that a warp's threads reach the barrier together; the callers come out of loops whose
    length differs by lane."""
    assert re.findall(r"barrier\.cluster\.\w+\.\w+(\.aligned)?;", source("greedy.cu")) == ["", ""]
