"""What a call can do without it does without: a graph loaded with a budget uses no optional memory, and a
graph without one, on a device allocator that refuses beyond what that graph's call took, gives the same
results. Memory is counted in the bytes asked of the caller's allocator."""
import numpy as np
import pytest

from tests import gpu_cases as G

pytestmark = pytest.mark.gpu

ROOM = 1 << 40


@pytest.fixture(scope="module")
def H():
    import paper_2406_01911_gb300 as H
    H.lib()
    return H


class Meter:
    """Counts the live bytes of a device allocator and refuses what would take them past `cap`."""

    def __init__(self, H):
        import torch
        self.live, self.peak, self.cap, self.size = 0, 0, None, {}

        def alloc(nbytes, stream):
            if self.cap is not None and self.live + nbytes > self.cap:
                return 0
            p = torch.cuda.caching_allocator_alloc(nbytes, 0, stream)
            self.size[p] = nbytes
            self.live += nbytes
            self.peak = max(self.peak, self.live)
            return p

        def free(p, stream):
            self.live -= self.size.pop(p)
            torch.cuda.caching_allocator_delete(p)

        self.allocator = H.DeviceAllocator(alloc, free)

    def need(self, call):
        """(what call() returns, the bytes it took beyond those live before)."""
        self.peak = before = self.live
        out = call()
        return out, self.peak - before


def twins(H, n, hes, model="uniform_pair", p=0.05):
    """The same graph twice: without a budget, and with one that never binds."""
    out = []
    for budget in (0, ROOM):
        m = Meter(H)
        out.append((H.Graph(n, *G.csr(hes), model, int(p * G.P32), seed=3, hbm_budget_bytes=budget, allocator=m.allocator), m))
    return out


@pytest.mark.parametrize("theta", [40, 4000, 60_000])
@pytest.mark.parametrize("upper", ["closed", "prefix"])
def test_greedy_without_numbers(H, theta, upper):
    """One block, one cluster, a grid: picks and bounds by number and by id, chosen and for want of memory."""
    n, hes = G.random_graph(6, 3000, 2600, 9)
    (a, ma), (b, mb) = twins(H, n, hes, p=0.2)
    pa, pb = (g.pool(tag=0, roots="stratified").sample(theta) for g in (a, b))
    want, res = a.select_seeds(pa, None, 25, mode="fixed", upper=upper)
    (lean, rlean), need = mb.need(lambda: b.select_seeds(pb, None, 25, mode="fixed", upper=upper))
    ma.cap = ma.live + need
    tight, rtight = a.select_seeds(pa, None, 25, mode="fixed", upper=upper)
    for s, r in ((lean, rlean), (tight, rtight)):
        assert s.tolist() == want.tolist() and r["lambda_r1"].tolist() == res["lambda_r1"].tolist()
        assert r["upper"] == res["upper"]


def same_sets(pa, pb):
    sa, sb = G.gpu_sets(pa), G.gpu_sets(pb)
    return sa[0] == sb[0] and np.array_equal(sa[1], sb[1]) and np.array_equal(sa[2], sb[2])


@pytest.mark.parametrize("strategy", ["paper", "binomial_only", "lt"])
@pytest.mark.parametrize("arena", [0, 1])
def test_growth_without_optional_memory(H, strategy, arena):
    """Two growth steps (arena = 1: most sets built again by a repair launch), then a query, each on as much
    memory as a graph takes that keeps nothing."""
    n, hes = G.hub_graph(n=6000, hub_edges=40, hub_size=120, mid_edges=8, mid_size=200, m_rest=2500)
    (a, ma), (b, mb) = twins(H, n, hes, p=0.03)
    for g in (a, b) if arena else ():
        g.set_tuning(arena_entries_per_set=arena)
    pa, pb = (g.pool(tag=0, roots="stratified", strategy=strategy) for g in (a, b))
    for theta in (300, 900):
        _, need = mb.need(lambda: pb.sample(theta))
        ma.cap = ma.live + need
        pa.sample(theta)
        ma.cap = None
        assert same_sets(pa, pb)

    def query(g):
        g.set_schedule("plain")  # growing ahead follows measured times, and the bytes taken with it
        return g.select_seeds(g.pool(1, "stratified", strategy), g.pool(2, "stratified", strategy), 5, mode="brr", eps=0.4)

    (sb, rb), need = mb.need(lambda: query(b))
    ma.cap = ma.live + need
    sa, ra = query(a)
    assert sa.tolist() == sb.tolist() and ra["lambda_r1"].tolist() == rb["lambda_r1"].tolist()


@pytest.mark.parametrize("strategy", ["paper", "binomial_only"])
@pytest.mark.parametrize("arena", [0, 1])
def test_batch_without_optional_memory(H, strategy, arena):
    n, hes = G.random_graph(3, 2000, 1500, 9)
    (a, ma), (b, mb) = twins(H, n, hes, p=0.08)

    def batch(g):
        # the batch takes pools by their handles' addresses, and the bytes it needs follow that order
        made = []
        for tag in range(4):
            made.append(g.pool(tag, "stratified", strategy))
            while tag and made[-1].handle.value < pools[-1].handle.value:
                made.append(g.pool(tag, "stratified", strategy))
            pools = made[:1] if tag == 0 else [*pools, made[-1]]
        g.set_tuning(arena_entries_per_set=arena)
        out = H.hyperim_select_seeds_batch([(g, pools[0], pools[1], 3, 0.3, 1.0), (g, pools[2], pools[3], 9, 0.3, 1.0)])
        return [(s.tolist(), r["theta"], r["lambda_r1"].tolist(), r["lambda_r2"].tolist()) for s, r in out]

    want, need = mb.need(lambda: batch(b))
    ma.cap = ma.live + need
    assert batch(a) == want


@pytest.mark.parametrize("name", ["chunks", "short"])
def test_load_without_optional_memory(H, name):
    """Neighbourhoods with a chunk index and its eighths, then sets in as much memory as a graph without them
    takes; hyperedges of 5 to 16 members, whose directories are left out too when they have no room."""
    n, hes = {"chunks": lambda: G.layered_hub_graph(n=12000, groups=8, size=90, m_rest=3000),
              "short": lambda: (4000, [list(range(i, i + 9)) for i in range(3900)])}[name]()
    lists = G.csr(hes)
    mb = Meter(H)
    b, need = mb.need(lambda: H.Graph(n, *lists, "wc", 0, seed=3, hbm_budget_bytes=ROOM, allocator=mb.allocator))
    ma = Meter(H)
    ma.cap = need
    a = H.Graph(n, *lists, "wc", 0, seed=3, allocator=ma.allocator)
    for key, value in b.profile().items():
        assert np.array_equal(a.profile()[key], value), key
    (a, ma), (b, mb) = twins(H, n, hes, "wc")
    extra = ma.live - mb.live - 16 * a.stats()["index_entries"]  # directories, once loaded, stay
    pa, pb = a.pool(tag=0, roots="plain"), b.pool(tag=0, roots="plain")
    _, need = mb.need(lambda: pb.sample(20_000))
    ma.cap = mb.live + need + extra
    pa.sample(20_000)
    assert same_sets(pa, pb)


def test_forward_without_a_second_block(H):
    """A hub whose hyperedges hold 200 times n members: the blocks beyond one per SM take no more than their
    queues, and the counts are the same without them, under a budget or for want of memory."""
    import torch
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    n, rng = 5000, np.random.default_rng(8)
    hes = [[0] + rng.choice(n - 1, size=2500, replace=False).tolist() for _ in range(400)]
    (a, ma), (b, mb) = twins(H, n, hes, p=0.0005)
    live = ma.live
    (want, _, _), more = ma.need(lambda: a.forward_spread([1, 2, 3], 2 * sm + 90, seed=4))
    (lean, _, _), need = mb.need(lambda: b.forward_spread([1, 2, 3], 2 * sm + 90, seed=4))
    assert more - need <= sm * 4 * n and ma.live - live <= 2 * sm * 4 * n
    (a, ma), _ = twins(H, n, hes, p=0.0005)
    ma.cap = ma.live + need
    tight, _, _ = a.forward_spread([1, 2, 3], 2 * sm + 90, seed=4)
    assert lean.tolist() == want.tolist() == tight.tolist()
