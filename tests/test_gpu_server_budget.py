"""What a server's budget counts: the memory its graphs need, not what their loads and its workers could do
without."""
import pytest

from tests import gpu_cases as G

pytestmark = pytest.mark.gpu

ROOM = 1 << 40


def serve(H, budget, optional):
    """Three queries on two graphs, each growing its pools; optional: the graphs' loads take optional memory."""
    graphs = []
    for seed in (1, 2):
        n, hes = G.layered_hub_graph(seed, n=12000, groups=8, size=90, m_rest=3000)
        graphs.append(H.Graph(n, *G.csr(hes), "uniform_pair", int(0.03 * G.P32), seed=3,
                              hbm_budget_bytes=0 if optional else ROOM))
        graphs[-1].set_schedule("plain")  # growing ahead follows measured times, and the bytes held with it
    srv = H.Server(workers=1, hbm_budget_bytes=budget)
    ids = [srv.add_graph(g) for g in graphs]
    out = [srv.wait(srv.submit(ids[i], 5, eps)) for i, eps in ((0, 0.4), (1, 0.4), (0, 0.1))]
    assert all(r["status"] == 0 for _, r in out)
    stats = srv.stats()
    srv.close()
    for g in graphs:
        g.close()
    return [(s.tolist(), r["lambda_r2"].tolist()) for s, r in out], stats["evictions"], stats["device_bytes"]


def test_budget_counts_needed_memory():
    import paper_2406_01911_gb300 as H
    want, _, free = serve(H, 0, True)
    got, none, roomy = serve(H, ROOM, True)
    assert got == want and none == 0
    assert roomy < free  # the worker kept no neighbourhoods
    _, _, lean = serve(H, ROOM, False)
    assert lean < roomy  # the graphs took optional memory
    # the least budget without an eviction for graphs that took none, to a tenth of what they took
    lo, hi = lean // 8, 4 * lean
    while hi - lo > (roomy - lean) // 10:
        mid = (lo + hi) // 2
        if serve(H, mid, False)[1]:
            lo = mid
        else:
            hi = mid
    got, evictions, _ = serve(H, hi, True)
    assert got == want and evictions == 0
    got, evictions, _ = serve(H, lo - (hi - lo), True)
    assert got == want and evictions > 0
