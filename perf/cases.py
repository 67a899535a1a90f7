"""The work that users of this library have it do, as calls that can be timed and compared.

Every case goes through the public entry points of ``paper_2406_01911_gb300``. The hypergraphs are
those of the repository's own workloads (Zipf or uniform hyperedge sizes, preferential or uniform
membership), generated on the GPU from a seed, over the range from 1,000 to 2,000,000 vertices.

Kinds of call:

  query     a whole HyperIM_BRR query on fresh pools (``select_seeds(mode="brr")``), on a resident
            graph or, with ``load``, from the hyperedge lists on, and the coverage score of every
            vertex on the sets that its last round read
  fixed     a pool of a given number of RR sets, seed selection on it and the scores
  sample    a pool of a given number of RR sets and the scores: a rank's step of the sharded path
  select    seed selection, the spread estimate and the scores on pools that are there already
  load      the graph load and its layer profile, copied out
  coverage  the coverage count that allocates nothing, on RR sets the caller holds
  forward   forward Monte-Carlo influence of a seed set
  batch     many queries on many graphs in one call
  serve     a server's life: graphs registered, queries submitted, all results waited for

The scores (Eq. 2: the weight of the RR sets that hold a vertex, for all n vertices) are what the
sets come down to for whoever picks seeds; with the seeds come the coverages, the bounds and every
round's alpha. Outputs of a case have one shape whatever the seed: lists of varying length are
padded with zeros.
"""
import math

import numpy as np
import torch

import paper_2406_01911_gb300 as H

P32 = 1 << 32


def listed():
    return [
        # the smallest configuration, as a test or a notebook runs it: launches and latency count
        dict(name="tiny_fixed", kind="fixed", n=1000, m=500, law="uniform", hi=6, alpha=0.0, members="uniform",
             model="uniform_pair", p=0.05, roots="plain", strategy="paper", theta=10000, k=10),
        # a graph of the batched configuration's middle size is loaded and its layer profile read
        # out: what a service does when a new hypergraph arrives
        dict(name="load_14k", kind="load", n=14142, m=9192, law="zipf", hi=300, alpha=2.1, members="preferential",
             model="wc", p=0.0),
        # the 100k-vertex configuration, one probability for every pair (the cascade is
        # supercritical: half of the RR sets hold a third of the graph)
        dict(name="query_100k_uniform", kind="query", load=True, n=100_000, m=50_000, law="zipf", hi=200, alpha=2.1,
             members="preferential", model="uniform_pair", p=0.01, roots="stratified", strategy="paper",
             upper="closed", k=50, eps=0.1),
        # the 2M-vertex configuration of the benchmark, weighted cascade: hubs, mostly tiny sets
        dict(name="query_2m_wc", kind="query", load=True, n=2_000_000, m=1_000_000, law="zipf", hi=1000, alpha=1.9,
             members="preferential", model="wc", p=0.0, roots="stratified", strategy="paper", upper="closed",
             k=100, eps=0.1),
        # RR sets of the LT cascade on that graph: every set is one path
        dict(name="sample_2m_lt", kind="sample", n=2_000_000, m=1_000_000, law="zipf", hi=1000, alpha=1.9,
             members="preferential", model="wc", p=0.0, roots="stratified", strategy="lt", theta=10000),
        # the paper's own layer probabilities on a resident graph, a query as an analyst repeats it
        dict(name="query_100k_paper", kind="query", load=False, n=100_000, m=50_000, law="zipf", hi=200, alpha=2.1,
             members="preferential", model="paper_layer", p=0.0, roots="stratified", strategy="paper",
             upper="closed", k=50, eps=0.1),
        # the tighter stopping bound, plain roots and the Binomial strategy (exact IC semantics)
        dict(name="query_200k_prefix", kind="query", load=False, n=200_000, m=120_000, law="zipf", hi=300, alpha=2.1,
             members="preferential", model="wc", p=0.0, roots="plain", strategy="binomial_only", upper="prefix",
             k=50, eps=0.1),
        # a large budget chosen on pools that are kept: the greedy and the estimate alone
        dict(name="select_2m", kind="select", n=2_000_000, m=1_000_000, law="zipf", hi=1000, alpha=1.9,
             members="preferential", model="wc", p=0.0, roots="stratified", strategy="paper", theta=40000, k=200),
        # a serving loop's coverage check on RR sets it holds in its own memory
        dict(name="coverage_200k_sets", kind="coverage", n=2_000_000, sets=200_000, mean=30, k=100),
        # the independent check of a seed set by forward simulation
        dict(name="forward_100k", kind="forward", n=100_000, m=50_000, law="zipf", hi=200, alpha=2.1,
             members="preferential", model="uniform_pair", p=0.01, k=50, sims=256),
        # graphs of uneven size queried with three budgets each, in one call
        dict(name="batch_12_graphs", kind="batch", graphs=12, n_lo=1000, n_hi=200_000, hi=300, alpha=2.1, eps=0.1),
        # a server over resident graphs and a burst of queries
        dict(name="serve_3_graphs", kind="serve", graphs=3, n_lo=100_000, n_hi=1_000_000, hi=500, alpha=2.0,
             workers=4, queries=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, n_lo, n_hi, hi_top):
    n = _log(rng, n_lo, n_hi)
    ratio = rng.uniform(0.3, 1.0) if n <= 200_000 else rng.uniform(0.3, 0.5)
    hi = _log(rng, 6, hi_top)
    law = rng.choice(["zipf", "zipf", "zipf", "uniform"]) if hi <= 12 else "zipf"
    return dict(n=n, m=max(2, int(n * ratio)), law=law, hi=hi, alpha=round(rng.uniform(1.9, 2.1), 3),
                members=rng.choice(["preferential", "preferential", "uniform"]))


def _any_model(rng, n_hi=2_000_000):
    """A graph shape with an activation model whose cascades stay within the listed cases' cost."""
    model = rng.choice(["wc", "wc", "uniform_pair", "paper_layer"])
    if model == "wc":
        c = dict(_shape(rng, 1000, n_hi, 1000), model=model, p=0.0)
    elif model == "paper_layer":
        c = dict(_shape(rng, 1000, min(n_hi, 100_000), 200), model=model, p=0.0)
    else:
        c = dict(_shape(rng, 1000, min(n_hi, 60_000), 150), model=model)
        top = 0.05 if c["n"] <= 4000 else 0.01
        c["p"] = round(math.exp(rng.uniform(math.log(0.002), math.log(top))), 5)
    return c


def draw(rng):
    kind = rng.choice(["query", "query", "query", "fixed", "sample", "sample", "select", "load", "load", "coverage",
                       "forward", "batch", "serve"])
    roots = rng.choice(["stratified", "stratified", "plain"])
    strategy = rng.choice(["paper", "paper", "binomial_only"])
    if kind == "query":
        return dict(_any_model(rng), kind=kind, load=rng.random() < 0.5, roots=roots, strategy=strategy,
                    upper=rng.choice(["closed", "closed", "closed", "prefix"]), k=_log(rng, 10, 200),
                    eps=rng.choice([0.1, 0.2]))
    if kind == "fixed":
        return dict(_any_model(rng, 60_000), kind=kind, roots=roots, strategy=strategy, theta=_log(rng, 200, 4000),
                    k=_log(rng, 1, 100))
    if kind == "sample":
        if rng.random() < 0.5:
            return dict(_shape(rng, 1000, 2_000_000, 1000), model="wc", p=0.0, kind=kind, roots=roots, strategy="lt",
                        theta=_log(rng, 200, 10000))
        return dict(_any_model(rng), kind=kind, roots=roots, strategy=strategy, theta=_log(rng, 100, 4000))
    if kind == "select":
        return dict(_shape(rng, 10_000, 2_000_000, 1000), model="wc", p=0.0, kind=kind, roots=roots,
                    strategy="paper", theta=_log(rng, 1000, 40000), k=_log(rng, 1, 200))
    if kind == "load":
        c = _any_model(rng, 200_000)
        return dict(c, kind=kind)
    if kind == "coverage":
        return dict(kind=kind, n=_log(rng, 1000, 4_000_000), sets=_log(rng, 1000, 200_000), mean=_log(rng, 2, 60),
                    k=_log(rng, 1, 200))
    if kind == "forward":
        return dict(_shape(rng, 1000, 60_000, 150), model="uniform_pair", p=0.01, kind=kind, k=_log(rng, 1, 100),
                    sims=_log(rng, 16, 256))
    if kind == "batch":
        return dict(kind=kind, graphs=rng.randint(2, 12), n_lo=1000, n_hi=_log(rng, 2000, 200_000), hi=300,
                    alpha=round(rng.uniform(2.0, 2.1), 3), eps=rng.choice([0.1, 0.2]))
    return dict(kind=kind, graphs=rng.randint(1, 3), n_lo=50_000, n_hi=_log(rng, 60_000, 1_000_000), hi=500,
                alpha=2.0, workers=rng.randint(1, 6), queries=rng.randint(2, 8))


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------
def _generator(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + salt) & 0x7FFFFFFFFFFFFFFF)
    return g


def _rand(gen, count):
    return torch.rand(count, generator=gen, device="cuda", dtype=torch.float64)


def _hyperedges(c, seed):
    """Hyperedge lists (offsets, members; int32 on the GPU): sizes uniform in [2, hi] or Zipf(alpha)
    truncated to it (the m quantiles of that law in random order); members uniform, or Chung-Lu
    with exponent 2.5 and the smallest power-of-two offset that keeps the largest expected degree
    below sqrt(nnz). A member may repeat."""
    gen = _generator(seed, 17)
    n, m, hi = c["n"], c["m"], min(c["hi"], c["n"])
    lo = min(2, hi)
    s = torch.arange(lo, hi + 1, device="cuda", dtype=torch.float64)
    pmf = torch.ones_like(s) if c["law"] == "uniform" else s ** (-c["alpha"])
    cdf = torch.cumsum(pmf / pmf.sum(), 0)
    quantile = (torch.randperm(m, generator=gen, device="cuda") + 0.5) / m
    sizes = lo + torch.searchsorted(cdf, quantile.double(), right=True).clamp_(max=hi - lo)
    off = torch.zeros(m + 1, device="cuda", dtype=torch.int64)
    torch.cumsum(sizes, 0, out=off[1:])
    nnz = int(off[-1])
    u = _rand(gen, nnz)
    if c["members"] == "uniform":
        mem = (u * n).to(torch.int64).clamp_(max=n - 1)
    else:
        v = torch.arange(n, device="cuda", dtype=torch.float64)
        i0 = 1
        while True:
            w = (v + i0) ** (-1.0 / 1.5)
            total = w.sum()
            if nnz * float(w[0] / total) <= math.sqrt(nnz) or i0 > n:
                break
            i0 *= 2
        mem = torch.searchsorted(torch.cumsum(w / total, 0), u, right=True).clamp_(max=n - 1)
    ids = torch.randperm(n, generator=gen, device="cuda")
    return off.to(torch.int32), ids[mem].to(torch.int32)


def _threshold(c):
    return int(c["p"] * P32)


def _load(c, seed, lists=None):
    off, mem = lists if lists is not None else _hyperedges(c, seed)
    return H.Graph(c["n"], off, mem, c["model"], _threshold(c), seed=seed & 0xFFFFFFFF)


def _some_graphs(c, seed):
    """`graphs` resident weighted-cascade hypergraphs, n spread evenly in the logarithm."""
    out = []
    for i in range(c["graphs"]):
        t = i / max(c["graphs"] - 1, 1)
        n = int(round(c["n_lo"] * (c["n_hi"] / c["n_lo"]) ** t))
        ratio = (0.3, 0.65, 1.0)[i % 3] if c["kind"] == "batch" else 0.6
        spec = dict(n=n, m=max(2, int(n * ratio)), law="zipf", hi=c["hi"], alpha=c["alpha"], members="preferential",
                    model="wc", p=0.0)
        out.append(_load(spec, seed * 64 + i))
    return out


def _seed_set(n, k, seed):
    gen = _generator(seed, 29)
    return torch.randperm(n, generator=gen, device="cuda")[:k].to(torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": seed}
    if kind == "coverage":
        gen = _generator(seed, 41)
        # set sizes as RR pools have them: most hold a member or two, a few hold hundreds
        u = _rand(gen, case["sets"])
        sizes = (1.0 + 0.5 * (1.0 - u) ** (-0.7)).clamp_(max=50.0 * case["mean"])
        sizes = (sizes * (case["mean"] / sizes.mean())).to(torch.int64).clamp_(min=1)
        off = torch.zeros(case["sets"] + 1, device="cuda", dtype=torch.int64)
        torch.cumsum(sizes, 0, out=off[1:])
        st["off"] = off
        st["mem"] = (_rand(gen, int(off[-1])) ** 3 * case["n"]).to(torch.int32).clamp_(max=case["n"] - 1)
        st["stratum"] = (_rand(gen, case["sets"]) * H.NSTRATA).to(torch.uint8).clamp_(max=H.NSTRATA - 1)
        st["seeds"] = (_rand(gen, case["k"]) ** 3 * case["n"]).to(torch.int32).clamp_(max=case["n"] - 1)
        return st
    if kind in ("batch", "serve"):
        st["graphs"] = _some_graphs(case, seed)
        if kind == "serve":
            # a burst over all graphs, budgets over the served range [10, 200]
            st["queries"] = [(i % case["graphs"], 10 + 53 * i % 191, (0.1, 0.2)[i // 3 % 2])
                             for i in range(case["queries"])]
        return st
    lists = _hyperedges(case, seed)
    if kind == "load" or case.get("load"):
        st["lists"] = lists
        return st
    g = _load(case, seed, lists)
    st["graph"] = g
    if kind == "select":
        st["r1"] = g.pool(0, case["roots"], case["strategy"]).sample(case["theta"])
        st["r2"] = g.pool(1, case["roots"], case["strategy"]).sample(case["theta"])
    if kind == "forward":
        st["seeds"] = _seed_set(case["n"], case["k"], seed).cpu().numpy()
    return st


# ------------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------------
def _scores(graph, pool, theta=0):
    """The coverage score of every vertex on the pool's sets (those of theta; 0: all of them)."""
    out = torch.empty(graph.n, device="cuda", dtype=torch.int64)
    rounds = H.GreedyRounds(graph, pool, theta)
    rounds.scores_into(out.data_ptr())
    rounds.end()
    return out


def _answers(pairs):
    """(seeds, result) of queries as three arrays: the seeds, the integers, the estimates and
    bounds with every round's alpha (64 places)."""
    ints = [x for _, r in pairs for x in (r["rounds"], r["theta"], r["pool_r1"], r["pool_r2"], *r["lambda_r1"].tolist(),
                                          *r["lambda_r2"].tolist())]
    reals = [x for _, r in pairs for x in (r["sigma_r1"], r["sigma_r2"], r["upper"], r["lower"], r["alpha"],
                                           *r["alpha_round"], *[0.0] * (64 - len(r["alpha_round"])))]
    return [np.concatenate([s for s, _ in pairs]), np.array(ints, np.int64), np.array(reals, np.float64)]


def _padded(profile, most):
    """A layer profile with its per-layer arrays as long as a profile can be (one per incidence)."""
    return {k: np.concatenate([a, np.zeros(most - len(a), a.dtype)]) if k.startswith("layer_") else a
            for k, a in profile.items()}


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "load":
        g = _load(c, state["seed"], state["lists"])
        return _padded(g.profile(), len(state["lists"][1]))
    if kind == "query":
        g = _load(c, state["seed"], state["lists"]) if c["load"] else state["graph"]
        r1, r2 = g.pool(0, c["roots"], c["strategy"]), g.pool(1, c["roots"], c["strategy"])
        seeds, res = g.select_seeds(r1, r2, c["k"], mode="brr", eps=c["eps"], upper=c["upper"])
        return _answers([(seeds, res)]) + [_scores(g, r1, res["theta"])]
    if kind == "fixed":
        g = state["graph"]
        pool = g.pool(0, c["roots"], c["strategy"]).sample(c["theta"])
        return _answers([g.select_seeds(pool, None, c["k"], mode="fixed")]) + [_scores(g, pool)]
    if kind == "sample":
        g = state["graph"]
        return [_scores(g, g.pool(0, c["roots"], c["strategy"]).sample(c["theta"]))]
    if kind == "select":
        g = state["graph"]
        seeds, res = g.select_seeds(state["r1"], state["r2"], c["k"], mode="fixed")
        sigma, err = g.spread(seeds, state["r2"])
        return _answers([(seeds, res)]) + [sigma, err, _scores(g, state["r1"])]
    if kind == "coverage":
        lam = torch.empty(H.NSTRATA, device="cuda", dtype=torch.int64)
        status = H.lib().hyperim_coverage_noalloc(
            c["n"], state["off"].data_ptr(), state["mem"].data_ptr(), state["stratum"].data_ptr(), c["sets"],
            state["seeds"].data_ptr(), c["k"], lam.data_ptr(), H.current_stream())
        return [lam, status]
    if kind == "forward":
        return list(state["graph"].forward_spread(state["seeds"], c["sims"], state["seed"]))
    if kind == "batch":
        queries = []
        for g in state["graphs"]:
            r1, r2 = g.pool(0, "stratified"), g.pool(1, "stratified")
            queries += [(g, r1, r2, k, c["eps"], 1.0) for k in (10, 50, 100)]
        return _answers(H.hyperim_select_seeds_batch(queries))
    server = H.Server(workers=c["workers"])
    ids = [server.add_graph(g) for g in state["graphs"]]
    tickets = [server.submit(ids[i], k, eps) for i, k, eps in state["queries"]]
    out = [server.wait(t) for t in tickets]
    server.close()
    return _answers(out) + [[r["status"] for _, r in out]]


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without, and 64-bit values
# ------------------------------------------------------------------------------------------------
def _incidences(n, m, law, hi, alpha):
    hi = min(hi, n)
    s = np.arange(min(2, hi), hi + 1, dtype=np.float64)
    pmf = np.ones_like(s) if law == "uniform" else s ** (-alpha)
    return m * float((s * pmf).sum() / pmf.sum())


def work(case):
    """Bytes: the hyperedge lists read once, the RR sets asked for written once (offset, stratum,
    index and at least the root), the outputs written once; pools that are there are read once."""
    kind = case["kind"]
    if kind == "coverage":
        return {"bytes": case["sets"] * (8 + 1 + 4.0 * case["mean"]) + 4.0 * case["k"] + 8.0 * H.NSTRATA, "flops": 0.0}
    if kind in ("batch", "serve"):
        total = 0.0
        for i in range(case["graphs"]):
            n = case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** (i / max(case["graphs"] - 1, 1))
            ratio = (0.3, 0.65, 1.0)[i % 3] if kind == "batch" else 0.6
            total += 4.0 * (_incidences(n, n * ratio, "zipf", case["hi"], case["alpha"]) + n * ratio)
        return {"bytes": total, "flops": 0.0}
    lists = 4.0 * (_incidences(case["n"], case["m"], case["law"], case["hi"], case["alpha"]) + case["m"] + 1)
    if kind == "load":
        return {"bytes": lists + case["n"] * (3 * 4.0 + 8.0), "flops": 0.0}
    if kind == "select":
        return {"bytes": 2 * 17.0 * case["theta"] + 4.0 * case["k"] + 8.0 * case["n"], "flops": 0.0}
    if kind == "forward":
        return {"bytes": lists + 4.0 * case["sims"], "flops": 0.0}
    return {"bytes": lists + 17.0 * case.get("theta", 0) + 4.0 * case.get("k", 0) + 8.0 * case["n"], "flops": 0.0}


def exact(case, seed):
    if case["kind"] == "coverage":
        st = prepare(case, seed)
        flag = torch.zeros(case["n"], device="cuda", dtype=torch.bool)
        flag[st["seeds"].long()] = True
        owner = torch.repeat_interleave(torch.arange(case["sets"], device="cuda"), st["off"].diff())
        hit = torch.zeros(case["sets"], device="cuda", dtype=torch.int64)
        hit[owner[flag[st["mem"].long()]]] = 1
        lam = torch.zeros(H.NSTRATA, device="cuda", dtype=torch.int64)
        lam.index_add_(0, st["stratum"].long(), hit)
        return [lam, 0]
    if case["kind"] == "load" and case["model"] != "paper_layer":
        # the layer profile from all ordered co-member pairs, counted
        n, m = case["n"], case["m"]
        off, mem = _hyperedges(case, seed)
        he = torch.repeat_interleave(torch.arange(m, device="cuda"), off.long().diff())
        key = torch.unique(he * n + mem.long())
        he, mem = key // n, key % n
        size = torch.bincount(he, minlength=m)
        start = torch.cumsum(size, 0) - size
        rows = torch.repeat_interleave(torch.arange(len(he), device="cuda"), size[he])
        first = torch.cumsum(size[he], 0) - size[he]
        other = mem[start[he[rows]] + torch.arange(len(rows), device="cuda") - first[rows]]
        u = mem[rows]
        pair, w = torch.unique((u * n + other)[u != other], return_counts=True)
        u = pair // n
        wmax = int(w.max()) + 1 if len(w) else 1
        layer, count = torch.unique(u * wmax + (wmax - 1 - w), return_counts=True)
        owner, lw = layer // wmax, wmax - 1 - layer % wmax
        deg = torch.bincount(u, minlength=n)
        nl = torch.bincount(owner, minlength=n)
        if case["model"] == "wc":
            thr = P32 // deg[owner].clamp(min=1)
        else:
            thr = torch.full_like(lw, _threshold(case))
        poff = torch.zeros(n + 1, device="cuda", dtype=torch.int64)
        torch.cumsum(nl, 0, out=poff[1:])
        pad = lambda x: torch.nn.functional.pad(x, (0, int(off[-1]) - len(x)))
        return {"deg": deg, "nlayers": nl, "stratum": nl.clamp(max=H.NSTRATA - 1), "prof_off": poff,
                "layer_w": pad(lw), "layer_n": pad(count), "layer_thr": pad(thr)}
    return None
