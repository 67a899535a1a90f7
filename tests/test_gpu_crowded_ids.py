"""Neighbourhoods crowded into few ids and many layers: thousands of chunks, most of them empty, counted a few
at a time. The index is the oracle's, sets drawn through it too, and loading takes about as long as with the
ids spread out."""
import time

import numpy as np
import pytest

from tests import gpu_cases as G
from tests.test_gpu_parity import check_chunk_index

pytestmark = pytest.mark.gpu


def crowd(hubs, layers, n, spread=False):
    """Every hub shares j + 1 hyperedges with the j-th id of a run of `layers` ids of its own."""
    ids = np.arange(n) if not spread else np.random.default_rng(1).permutation(n)
    return n, [[int(ids[n - 1 - h])] + [int(ids[h * layers + x]) for x in range(j, layers)]
               for h in range(hubs) for j in range(layers)]


@pytest.mark.parametrize("hubs,layers,n", [(2, 60, 8192), (1, 100, 4096), (1, 127, 130), (2, 120, 8192)])
def test_crowded_index_equals_oracle(oracle, hubs, layers, n):
    import paper_2406_01911_gb300 as H
    n, hes = crowd(hubs, layers, n)
    off, mem = G.csr(hes)
    g = H.Graph(n, off, mem, "wc", 0, seed=9)
    og = oracle.Graph(n, off, mem, "wc", 0)
    assert check_chunk_index(g, og, n, [0, 1, layers // 2, layers - 1, n - 1]) > 0
    op = oracle.Pool(og, seed=9, tag=0, roots="stratified")
    op.grow_theta(300)
    G.assert_same_pool(g.pool(tag=0, roots="stratified").sample(300), op)


def test_crowded_load_time():
    import torch

    import paper_2406_01911_gb300 as H

    def seconds(spread):
        n, hes = crowd(6, 120, 8192, spread)
        lists = [torch.as_tensor(x, device="cuda") for x in G.csr(hes)]
        best = 1e9
        for _ in range(7):
            torch.cuda.synchronize()
            t = time.perf_counter()
            H.Graph(n, *lists, "wc", 0, seed=1).close()
            best = min(best, time.perf_counter() - t)
        return best

    # 76M index entries against 1M, graph freed again: 2.9 times as long, 8 times when every group of chunks
    # walked every key
    assert seconds(False) < 5 * seconds(True)
