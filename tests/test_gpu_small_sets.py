"""Sets that are small on average against the plain schedule (a block per set), one growth step on
either side of the number of sets from which single warps begin them (four for every warp)."""
import numpy as np
import pytest
import torch

from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("more", [-1, 0])
def test_small_sets_by_warps_equal_plain(more):
    import paper_2406_01911_gb300 as H
    steps = 64 * torch.cuda.get_device_properties(0).multi_processor_count + more
    rng = np.random.default_rng(4)
    off = np.arange(0, 478 * 6 + 1, 6, dtype=np.int32)
    g = H.Graph(1188, off, rng.integers(0, 1188, size=478 * 6, dtype=np.int32), "wc", 0, seed=5)
    got = G.gpu_sets(g.pool(tag=0, roots="plain").sample(100).sample(100 + steps))
    g.set_schedule("plain")
    want = G.gpu_sets(g.pool(tag=0, roots="plain").sample(100 + steps))
    assert got[0] == want[0] and np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])
