"""LT sets built one warp per set against the block-per-set kernel (the plain schedule), at the
sizes where the warp's member set and queue change: sets that never leave a tiny queue, sets past
the on-chip sort buffer (2,048 members) and sets past the queue (4,096: built again by a block)."""
import numpy as np
import pytest

from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    import paper_2406_01911_gb300 as H
    H.lib()
    return H


def uniform_graph(n, m, size, seed=3):
    """m hyperedges of `size` uniform members; one hyperedge of everybody when m = 1."""
    rng = np.random.default_rng(seed)
    off = np.arange(0, (m + 1) * size, size, dtype=np.int32)
    return off, np.arange(n, dtype=np.int32) if m == 1 else rng.integers(0, n, size=m * size, dtype=np.int32)


@pytest.mark.parametrize("n,m,size,theta,longest", [(2, 1, 2, 40, 2), (31, 40, 4, 300, 8), (33, 40, 4, 300, 8),
                                                    (4097, 1, 4097, 500, 100),
                                                    (3_000_000, 4500, 2000, 300, 4097)])
def test_lt_path_phase_equals_block_kernel(H, n, m, size, theta, longest):
    off, mem = uniform_graph(n, m, size)
    g = H.Graph(n, off, mem, "wc", 0, seed=5)
    got = G.gpu_sets(g.pool(tag=0, roots="stratified", strategy="lt").sample(theta // 3).sample(theta))
    g.set_schedule("plain")
    want = G.gpu_sets(g.pool(tag=0, roots="stratified", strategy="lt").sample(theta))
    assert got[0] == want[0] and np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])
    assert max(len(x) for x in want[0]) >= longest
