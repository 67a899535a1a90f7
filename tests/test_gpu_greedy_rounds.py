"""The one-launch greedy and the on-chip coverage at the sizes where they change: one block and many
(16,384 members a block), exhausted coverage, scores of one and of several radix digits, seed sets
around the 2,048 that a block holds. Reference: Alg. 1, Eq. 2 and Eq. upper_2 in Python integers over
the pool's sets."""
import ctypes as C

import numpy as np
import pytest

from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    import paper_2406_01911_gb300 as H
    H.lib()
    return H


def reference(n, sets, weights, k):
    """(seeds, covered sets per seed list, least Eq. upper_2 bound in weight units)."""
    score = [0] * n
    holds = [[] for _ in range(n)]
    for r, s in enumerate(sets):
        for v in s:
            score[v] += weights[r]
            holds[v].append(r)
    picked, covered, cover, best = [], set(), 0, None
    for i in range(k + 1):
        left = [score[v] for v in range(n) if v not in set(picked)]
        bound = cover + sum(sorted(left, reverse=True)[:k])
        best = bound if best is None else min(best, bound)
        if i == k:
            break
        v = min((u for u in range(n) if u not in set(picked)), key=lambda u: (-score[u], u))
        picked.append(v)
        cover += score[v]
        for r in holds[v]:
            if r not in covered:
                covered.add(r)
                for u in sets[r]:
                    score[u] -= weights[r]
    return picked, covered, best


@pytest.mark.parametrize("n,m,smax,theta,k", [(12, 8, 3, 30, 12), (90, 40, 6, 300, 90), (300, 200, 8, 700, 20),
                                              (600, 500, 10, 2600, 9), (600, 500, 10, 9000, 9)])
@pytest.mark.parametrize("roots", ["plain", "stratified"])
def test_greedy_rounds_and_prefix_bound(H, n, m, smax, theta, k, roots):
    n, hes = G.random_graph(5, n, m, smax)
    g = H.Graph(n, *G.csr(hes), "uniform_pair", int(0.15 * G.P32), seed=3)
    p = g.pool(tag=0, roots=roots).sample(theta)
    off, mem, st, _ = p.to_host()
    sets = [mem[off[r]:off[r + 1]].tolist() for r in range(len(off) - 1)]
    size, n_s = g.stats()["stratum_size"], p.view()["n_s"]
    w = [1] * len(sets) if roots == "plain" else [(size[s] << 32) // int(n_s[s]) for s in st.tolist()]
    seeds, covered, bound = reference(n, sets, w, k)
    got, res = g.select_seeds(p, None, k, mode="fixed", upper="prefix")
    assert got.tolist() == seeds
    lam = np.bincount(st[sorted(covered)], minlength=16)
    assert res["lambda_r1"].tolist() == lam.tolist()
    want = bound * (n / len(sets) if roots == "plain" else 2.0 ** -32)
    assert abs(res["upper"] - want) <= 1e-12 * want


@pytest.mark.parametrize("k", [0, 1, 2047, 2048, 2049])
@pytest.mark.parametrize("theta", [40, 20000])
def test_coverage_on_chip_and_with_flags(H, k, theta):
    import torch
    n, hes = G.random_graph(9, 5000, 3000, 9)
    g = H.Graph(n, *G.csr(hes), "uniform_pair", int(0.1 * G.P32), seed=4)
    p = g.pool(tag=0, roots="stratified").sample(theta)
    seeds = np.random.default_rng(k).integers(0, n, size=k).astype(np.int32)
    off, mem, st, j = p.to_host()
    hit = np.add.reduceat(np.isin(mem, seeds).astype(np.int64), off[:-1]) > 0
    want = np.bincount(st[hit], minlength=16)
    assert H.hyperim_coverage_view(g, p, 0, seeds).tolist() == want.tolist()
    # a prefix view: the sets of a smaller theta
    small = g.pool(tag=0, roots="stratified").sample(theta // 3)
    lim = small.view()["n_s"]
    inside = hit & (j < np.asarray(lim)[st])
    assert H.hyperim_coverage_view(g, p, theta // 3, seeds).tolist() == np.bincount(st[inside], minlength=16).tolist()
    v = p.view()
    lam = torch.full((16,), 7, dtype=torch.int64, device="cuda")
    sd = torch.as_tensor(seeds, device="cuda")
    assert H.lib().hyperim_coverage_noalloc(n, C.c_void_p(v["rr_off"]), C.c_void_p(v["rr_mem"]), C.c_void_p(v["rr_stratum"]),
                                            v["count"], C.c_void_p(sd.data_ptr() if k else None), k,
                                            C.c_void_p(lam.data_ptr()), C.c_void_p(H.current_stream())) == 0
    assert lam.tolist() == want.tolist()


@pytest.mark.parametrize("p,theta", [(0.02, 60000), (0.3, 30000), (0.9, 60), (0.9, 400)])
@pytest.mark.parametrize("roots", ["plain", "stratified"])
def test_candidates_give_the_stepwise_picks(H, p, theta, roots):
    """Enough vertices for candidates: scores that fall slowly, and (one giant component, p = 0.9) to
    nothing after the first picks, so that the candidates have to be chosen anew; pools of one cluster and
    of a grid. The stepwise greedy looks at every vertex in every round."""
    n, hes = G.random_graph(11, 60_000, 60_000, 5)
    g = H.Graph(n, *G.csr(hes), "uniform_pair", int(p * G.P32), seed=6)
    pool = g.pool(tag=0, roots=roots).sample(theta)
    k = 120
    seeds, res = g.select_seeds(pool, None, k, mode="fixed")
    rounds = H.GreedyRounds(g, pool)
    assert seeds.tolist() == [rounds.pick() for _ in range(k)]
    assert res["lambda_r1"].tolist() == rounds.end().tolist()
