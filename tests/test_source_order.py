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


def test_kept_neighbourhoods_are_published_and_acquired():
    """The entries are written, then the slot, after a fence of the thread that writes it; every read of a slot
    acquires, in the warp's pop for all lanes (a shuffle orders no memory)."""
    rr = source("rr.cu")
    readers = set(re.findall(r"(\w+)\(P\.memo_slot \+ mu\)", rr))
    assert len(readers) == 1
    assert re.search(r"%s\(const uint32_t\* p\) \{[^}]*ld\.acquire\.gpu" % readers.pop(), rr)
    publish = re.sub(r"\s+", " ", body(rr, "void memo_publish"))
    assert "__syncwarp();" in publish and publish.index("__syncwarp();") < publish.index("__threadfence();")
    assert re.search(r"__threadfence\(\);\s*atomicExch\(P\.memo_slot", publish)
    warp = re.sub(r"\s+", " ", body(rr, "bool pop_warp("))
    assert "kept = __shfl_sync(0xFFFFFFFFu, kept, 0); __syncwarp();" in warp
