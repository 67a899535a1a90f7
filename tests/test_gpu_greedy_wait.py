"""The greedy's grid (pools of more than 4M members) waits no longer than its handle's limit, and the handle
works on after a wait ran out; the Eq. upper_2 bound there."""
import numpy as np
import pytest

from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pool():
    import paper_2406_01911_gb300 as H
    n, hes = G.random_graph(11, 4000, 3000, 8)
    g = H.Graph(n, *G.csr(hes), "uniform_pair", int(0.3 * G.P32), seed=3)
    p = g.pool(tag=0, roots="stratified").sample(4000)
    assert p.view()["total"] > 1 << 22
    return H, g, p


def test_barrier_follows_the_wait_limit(pool):
    H, g, p = pool
    g.set_wait_limit(1)
    with pytest.raises(H.HyperIMError) as e:
        g.select_seeds(p, None, 20, mode="fixed")
    assert e.value.status == -4  # HYPERIM_ETIMEDOUT
    g.set_wait_limit(0)
    seeds, res = g.select_seeds(p, None, 20, mode="fixed")
    rounds = H.GreedyRounds(g, p)
    assert seeds.tolist() == [rounds.pick() for _ in range(20)]
    assert res["lambda_r1"].tolist() == rounds.end().tolist()


def test_prefix_bound_in_the_grid(pool):
    """Least over the rounds of the weight covered so far plus the k largest scores left, in whole numbers
    from the pool's sets."""
    H, g, p = pool
    k, n = 12, g.n
    off, mem, st, _ = p.to_host()
    size, n_s = g.stats()["stratum_size"], p.view()["n_s"]
    w = np.array([(size[s] << 32) // int(n_s[s]) for s in st], dtype=np.int64)
    owner = np.repeat(np.arange(len(st)), np.diff(off))
    left = np.ones(len(st), dtype=bool)
    best, cover, picked = None, 0, []
    for i in range(k + 1):
        part = left[owner]
        score = np.zeros(n, dtype=np.int64)
        np.add.at(score, mem[part], w[owner[part]])
        bound = cover + sum(int(x) for x in np.sort(score)[-k:])
        best = bound if best is None else min(best, bound)
        if i < k:
            v = int(np.argmax(score))
            picked.append(v)
            cover += int(score[v])
            left[owner[mem == v]] = False
    seeds, res = g.select_seeds(p, None, k, mode="fixed", upper="prefix")
    assert seeds.tolist() == picked
    want = best * 2.0 ** -32
    assert abs(res["upper"] - want) <= 1e-12 * want
