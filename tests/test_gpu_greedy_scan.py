"""Selection where nearly all scores are alike (sets of a member or two): no candidates to keep, round after
round, many vertices or few of them in a set."""
import time

import numpy as np
import pytest

from tests import gpu_cases as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def H():
    import paper_2406_01911_gb300 as H
    H.lib()
    return H


def graph(H, budget=0, n=2_000_000):
    mem = np.random.default_rng(2).integers(0, n, size=3 * (n // 2), dtype=np.int32)
    return H.Graph(n, np.arange(0, len(mem) + 1, 3, dtype=np.int32), mem, "uniform_pair", int(0.05 * G.P32), seed=3,
                   hbm_budget_bytes=budget)


def seconds(g, pool, k=100):
    best = 1e9
    for _ in range(5):
        t = time.perf_counter()
        g.select_seeds(pool, None, k, mode="fixed")
        best = min(best, time.perf_counter() - t)
    return best


def same_as_stepwise(H, g, pool, k=100):
    seeds, res = g.select_seeds(pool, None, k, mode="fixed")
    rounds = H.GreedyRounds(g, pool)
    return seeds.tolist() == [rounds.pick() for _ in range(k)] and res["lambda_r1"].tolist() == rounds.end().tolist()


def stepwise_seconds(H, g, pool, k=100):
    best = 1e9
    for _ in range(3):
        t = time.perf_counter()
        rounds = H.GreedyRounds(g, pool)
        for _ in range(k):
            rounds.pick()
        rounds.end()
        best = min(best, time.perf_counter() - t)
    return best


@pytest.mark.parametrize("theta", [40_000, 400_000])
def test_scores_alike(H, theta):
    g = graph(H)
    pool = g.pool(tag=0, roots="stratified").sample(theta)
    assert same_as_stepwise(H, g, pool)
    a, b = seconds(g, pool), stepwise_seconds(H, g, pool)
    assert a < b  # the stepwise form takes two launches and a wait of the host for every round


@pytest.mark.parametrize("n,theta", [(40_000, 500), (300_000, 3000), (600_000, 3000), (600_000, 60_000), (2_000_000, 3000)])
def test_few_members_without_numbers(H, n, theta):
    """Under a budget the vertices keep their ids, and a round may read every vertex's score."""
    g = graph(H, 1 << 40, n)
    pool = g.pool(tag=0, roots="stratified").sample(theta)
    assert same_as_stepwise(H, g, pool)
    assert seconds(g, pool) < stepwise_seconds(H, g, pool)
