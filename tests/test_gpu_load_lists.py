"""Graph load at the sizes where its list sorts, strata lists and layer histogram change: hyperedges and
vertex lists across the lanes (32), per warp (1,024), per block (8,192) and beyond, repeated members,
strata runs (512 vertices), more layers than the on-chip histogram holds (256)."""
import numpy as np
import pytest

from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    import paper_2406_01911_gb300 as H
    H.lib()
    return H


def sized(size, n):
    """A hyperedge of `size` entries in falling id order, one of them twice, among a few pairs."""
    rng = np.random.default_rng(size)
    he = sorted((int(x) for x in rng.choice(n, size=size - 1, replace=False)), reverse=True)
    return n, [[0, n - 1], he + [he[len(he) // 2]]] + [[int(x) for x in rng.integers(0, n, size=3)] for _ in range(40)]


def star(degree, n):
    """Vertex 0 in `degree` pairs, each other vertex in a few."""
    return n, [[1 + i % (n - 1), 0] for i in range(degree)]


def many_layers(layers):
    """Vertex 0 shares i hyperedges with vertex i: one layer each."""
    return layers + 2, [[0, *range(j, layers + 1)] for j in range(1, layers + 1)]


CASES = {**{f"he{s}": (lambda s=s: sized(s, max(2 * s, 600))) for s in (31, 32, 33, 1023, 1024, 1025, 8191, 8192, 8193)},
         **{f"v{d}": (lambda d=d: star(d, 90)) for d in (32, 33, 1024, 1025, 8192, 8193)},
         **{f"n{n}": (lambda n=n: G.random_graph(n, n, n, 5)) for n in (1, 511, 512, 513, 1025)},
         **{f"l{x}": (lambda x=x: many_layers(x)) for x in (254, 256, 257)}}


@pytest.mark.parametrize("name", sorted(CASES))
def test_load_lists(H, oracle, name):
    n, hes = CASES[name]()
    off, mem = G.csr(hes)
    g = H.Graph(n, off, mem, "paper_layer", 0, seed=5)
    og = oracle.Graph(n, off, mem, "paper_layer", 0)
    a = g.profile()
    for v in sorted({0, n // 2, n - 1} | set(range(0, n, max(1, n // 60))) | set(hes[0])):
        b, e = a["prof_off"][v], a["prof_off"][v + 1]
        got = list(zip(a["layer_w"][b:e].tolist(), a["layer_n"][b:e].tolist(), a["layer_thr"][b:e].tolist()))
        assert got == [tuple(int(x) for x in t) for t in og.layers(v)], v
        assert (a["deg"][v], a["nlayers"][v], a["stratum"][v]) == (og.deg(v), og.nlayers(v), og.stratum(v)), v
    # the strata lists, through the roots they give
    pool, op = g.pool(tag=0, roots="stratified").sample(20), oracle.Pool(og, seed=5, tag=0, roots="stratified")
    op.grow_theta(20)
    G.assert_same_pool(pool, op)
