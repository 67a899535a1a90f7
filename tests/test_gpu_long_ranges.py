"""Neighbourhoods read in id ranges that hold more than 16 members of a hyperedge: few and many hyperedges,
around the 32 and 128 of a group, long and short ranges side by side, with and without directories."""
import numpy as np
import pytest

from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,size", [(3, 3000), (31, 900), (33, 400), (33, 120), (127, 150), (130, 40)])
@pytest.mark.parametrize("budget", [0, 1 << 40])
def test_long_ranges_equal_oracle(oracle, count, size, budget):
    import paper_2406_01911_gb300 as H
    n, rng = 4000, np.random.default_rng(count)
    hes = [[0, *rng.choice(np.arange(1, n), size=size - 1, replace=False).tolist()] for _ in range(count)]
    # a hyperedge of 2,000 neighbouring ids makes one range of each vertex long, pairs make the others short
    hes += [[0, *range(1000, 3000)]] + [[0, int(v)] for v in rng.integers(1, n, size=20)]
    off, mem = G.csr(hes)
    og = oracle.Graph(n, off, mem, "paper_layer", 0)
    g = H.Graph(n, off, mem, "paper_layer", 0, seed=9, hbm_budget_bytes=budget)
    counts, _, _ = g.forward_spread([0, 5], 6, seed=2)
    assert counts.tolist() == og.forward_spread([0, 5], 6, seed=2).tolist()
    ow = oracle.Graph(n, off, mem, "wc", 0)
    w = H.Graph(n, off, mem, "wc", 0, seed=9, hbm_budget_bytes=budget)
    for strategy in ("paper", "lt"):
        op = oracle.Pool(ow, seed=9, tag=0, roots="stratified", strategy=strategy)
        op.grow_theta(60)
        G.assert_same_pool(w.pool(tag=0, roots="stratified", strategy=strategy).sample(60), op)
