"""Performance cases: what a user of the library has it do, through the Python binding.

A case is one kind of call (queries one by one, a batch of candidates, a mining run, a map count,
exact maximum independent sets, a graph load, a stream of served requests) on one data graph.  Graphs are seeded random graphs of the shapes the tests and the
benchmark use: Erdos-Renyi with uniform labels, or Chung-Lu (exponent 2.3) with Zipf labels,
undirected, directed or edge-labelled.  Patterns are random trees, paths, stars, cycles and
cliques whose vertex labels follow the graph's label distribution.  Everything is drawn from the
seed, graph and patterns alike.
"""
import itertools
import time

import numpy as np
import torch

import paper_2404_01585_gb300 as fx

MODES = {
    "early": fx.FLEXIS_MODE_EARLY,  # capped mIS and MNI
    "decide": fx.FLEXIS_MODE_EARLY | fx.FLEXIS_MODE_NO_MNI,  # mIS decision only
    "full": fx.FLEXIS_MODE_FULL,  # exact mIS and MNI
    "count": fx.FLEXIS_MODE_FULL | fx.FLEXIS_MODE_NO_MIS | fx.FLEXIS_MODE_COUNT_MAPS,  # |M| and exact MNI
    "exact_mis": fx.FLEXIS_MODE_FULL | fx.FLEXIS_MODE_NO_MNI | fx.FLEXIS_MODE_EXACT_MIS,
}
SHAPES = ("tree", "path", "star", "cycle", "clique")
FIELDS = ("status", "n", "sigma", "tau", "cap", "mis", "mni", "frequent", "flags", "n_maps", "mis_exact")
# the graph shapes of the workloads: Citeseer-, MiCo-, 1M-vertex-, YouTube-like
CITESEER = dict(law="er", nv=3312, ne=4732, nl=6)
MICO = dict(law="cl", nv=100_000, ne=1_080_000, nl=29, zipf=1.2)
CL1M = dict(law="cl", nv=1_000_000, ne=10_000_000, nl=37, zipf=1.0)
YOUTUBE = dict(law="cl", nv=4_600_000, ne=43_900_000, nl=80, zipf=1.0)


def listed():
    return [
        # one small interactive query: the smallest call, all latency
        dict(CITESEER, name="query citeseer", kind="query", count=1, nmin=3, nmax=5, sigma=30, lam=0.5,
             mode="full", acyclic=1),
        # an analyst's session of exact queries (mIS and MNI to the end), one after another
        dict(MICO, name="queries mico full", kind="query", count=8, nmin=3, nmax=5, sigma=1000, lam=0.5, mode="full"),
        # one level's candidates of a caller's own miner, medium graph
        dict(MICO, name="batch mico", kind="batch", count=256, nmin=3, nmax=6, sigma=1000, lam=0.5, mode="decide"),
        # the same on a 1M-vertex graph
        dict(CL1M, name="batch 1M", kind="batch", count=500, nmin=3, nmax=6, sigma=1000, lam=0.5, mode="decide"),
        # directed graph, directed patterns, capped mIS and MNI
        dict(law="cl", nv=20_000, ne=100_000, nl=6, zipf=1.0, name="batch directed", kind="batch", directed=1,
             count=200, nmin=3, nmax=5, sigma=200, lam=0.5, mode="early"),
        # mining a small graph deep: thousands of cheap candidates per level
        dict(CITESEER, name="mine citeseer", kind="mine", sigma=20, lam=0.5, edges=5, rows=1 << 14),
        # mining the MiCo-shaped graph: few heavy candidates
        dict(MICO, name="mine mico", kind="mine", sigma=3000, lam=0.5, edges=4, rows=1 << 12),
        # the same at lambda = 0, to 5 edges: a hundred thousand candidates, mostly frequent
        dict(MICO, name="mine mico deep", kind="mine", sigma=3000, lam=0.0, edges=5, rows=1 << 18),
        # count-only mode: every map counted, exact MNI
        dict(MICO, name="count mico", kind="batch", count=48, nmin=3, nmax=4, sigma=1000, lam=0.5, mode="count"),
        # maximum independent sets of small overlap graphs beside the greedy ones
        dict(law="er", nv=3000, ne=3300, nl=6, name="exact mis", kind="batch", count=32, nmin=3, nmax=4, sigma=60,
             lam=0.5, mode="exact_mis", nodes=4096),
        # a graph loaded from host arrays and its label pairs mined (the first level), then released
        dict(YOUTUBE, name="load youtube", kind="load", sigma=20_000, lam=0.5, edges=1, rows=1 << 12),
        # requests of mixed sizes and thresholds sent to a running server
        dict(MICO, name="serve mico", kind="serve", count=500, nmin=3, nmax=5, sigma=1000, lam=0.5, mode="decide",
             slots=256),
    ]


def _log(rng, lo, hi):
    return int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))


def draw(rng):
    kind = rng.choice(["query", "batch", "batch", "mine", "count", "exact_mis", "load", "serve"])
    c = dict(kind=kind, lam=rng.choice([0.0, 0.25, 0.5, 1.0]))
    if kind == "exact_mis":
        nv = _log(rng, 500, 4000)
        c.update(kind="batch", mode="exact_mis", law="er", nv=nv, ne=int(nv * rng.uniform(0.8, 1.2)),
                 nl=rng.randint(4, 10), count=rng.randint(4, 48), nmin=3, nmax=4, nodes=4096)
    else:
        nv = _log(rng, 2000, {"mine": 100_000, "count": 100_000, "load": 4_000_000}.get(kind, 1_000_000))
        if rng.random() < 0.3 and nv < 100_000:
            c.update(law="er", nv=nv, ne=int(nv * rng.uniform(1.2, 5.0)), nl=rng.randint(4, 12))
        else:
            c.update(law="cl", nv=nv, ne=int(nv * rng.uniform(2.0, 10.0)),
                     nl=rng.randint(6, 20) if nv < 50_000 else rng.randint(25, 80), zipf=rng.choice([1.0, 1.2]))
    c["sigma"] = max(4, int(c["nv"] * rng.uniform(0.01, 0.03)))
    if kind in ("mine", "load"):
        c["edges"] = 1 if kind == "load" else rng.randint(2, 4)
        c["rows"] = 1 << (12 if kind == "load" else 16)
        return c
    if kind in ("query", "batch"):
        form = rng.choice(["plain", "plain", "directed", "edge labels"])
        if form == "directed" and c["nv"] < 200_000:
            c["directed"] = 1
        elif form == "edge labels" and c["nv"] < 50_000:
            c["edge_labels"] = rng.randint(2, 5)
    if kind == "count":
        c.update(kind="batch", mode="count", count=rng.randint(1, 48), nmin=3, nmax=4)
    elif kind != "exact_mis":
        c.update(nmin=3, nmax=rng.randint(4, 5), mode=rng.choice(["early", "decide", "decide", "full"]),
                 count=rng.randint(1, 8) if kind == "query" else _log(rng, 9, 700))
        if c["nv"] > 200_000 and c["mode"] == "full":
            c["mode"] = "early"
    if c.get("edge_labels"):
        c["nmax"] = 4  # a pattern and its edges have at most 8 vertices between them
    if kind == "serve":
        c.update(mode="decide", slots=rng.choice([32, 256]), count=_log(rng, 20, 600))
    return c


# ---------------------------------------------------------------- inputs

def _cdf(w):
    c = np.cumsum(w)
    return c / c[-1]


def make_graph(c, seed):
    """(labels, src, dst, edge labels or None): host arrays; exactly ne distinct edges."""
    nv, ne = c["nv"], c["ne"]
    dev = "cuda"
    gen = torch.Generator(device=dev).manual_seed(seed)
    if c["law"] == "cl":
        # endpoint i proportional to (i + 1)^(-1 / (gamma - 1)), gamma = 2.3
        cdf = torch.from_numpy(_cdf(np.arange(1, nv + 1, dtype=np.float64) ** (-1.0 / 1.3))).to(dev)

        def ends(k):
            u = torch.rand(k, dtype=torch.float64, device=dev, generator=gen)
            return torch.searchsorted(cdf, u, right=True).clamp_(max=nv - 1)
    else:
        def ends(k):
            return torch.randint(0, nv, (k,), device=dev, generator=gen)
    keys = torch.empty(0, dtype=torch.int64, device=dev)
    while keys.numel() < ne:
        k = int((ne - keys.numel()) * 1.3) + 1024
        a, b = ends(k), ends(k)
        keys = torch.unique(torch.cat([keys, (torch.minimum(a, b) * nv + torch.maximum(a, b))[a != b]]))
    keys = keys[torch.randperm(keys.numel(), device=dev, generator=gen)[:ne]]
    perm = torch.randperm(nv, device=dev, generator=gen)
    src, dst = perm[keys // nv], perm[keys % nv]
    flip = torch.rand(ne, device=dev, generator=gen) < 0.5
    src, dst = torch.where(flip, dst, src), torch.where(flip, src, dst)
    rng = np.random.default_rng([seed, 1])
    if c.get("zipf"):
        p = _cdf(np.arange(1, c["nl"] + 1, dtype=np.float64) ** -c["zipf"])
        lab = np.minimum(np.searchsorted(p, rng.random(nv), side="right"), c["nl"] - 1)
    else:
        lab = rng.integers(0, c["nl"], nv)
    el = rng.integers(0, c["edge_labels"], ne).astype(np.int32) if c.get("edge_labels") else None
    return lab.astype(np.int32), src.int().cpu().numpy(), dst.int().cpu().numpy(), el


def _shape(shape, n, rng):
    if shape == "path":
        return [(i, i + 1) for i in range(n - 1)]
    if shape == "star":
        return [(0, i) for i in range(1, n)]
    if shape == "cycle":
        return [(i, (i + 1) % n) for i in range(n)]
    if shape == "clique":
        return list(itertools.combinations(range(n), 2))
    return [(int(rng.integers(i)), i) for i in range(1, n)]  # a random recursive tree


def make_patterns(c, lab, seed):
    """(labels, edges) or (labels, edges, edge labels) per pattern."""
    rng = np.random.default_rng([seed, 2])
    out = []
    for _ in range(c["count"]):
        n = int(rng.integers(c["nmin"], c["nmax"] + 1))
        e = _shape(SHAPES[rng.integers(3 if c.get("acyclic") else len(SHAPES))], n, rng)
        if c.get("edge_labels"):
            e = e[:8 - n]
            n = max(max(x) for x in e) + 1
        if c.get("directed"):
            e = [(b, a) if rng.random() < 0.5 else (a, b) for a, b in e]
        p = (lab[rng.integers(0, c["nv"], n)], np.asarray(e, np.int32))
        if c.get("edge_labels"):
            p += (rng.integers(0, c["edge_labels"], len(e)).astype(np.int32),)
        out.append(p)
    return out


class State:
    def __init__(self, case, seed):
        c = self.case = case
        self.server = self.graph = None
        lab, src, dst, el = self.arrays = make_graph(c, seed)
        self.options = {k: v for k, v in (("directed", c.get("directed")), ("exact_mis_nodes", c.get("nodes"))) if v}
        if c["kind"] == "load":
            return
        self.graph = fx.Graph(lab, src, dst, edge_labels=el, **self.options)
        if c["kind"] == "mine":
            return
        self.mode = MODES[c["mode"]]
        self.patterns = make_patterns(c, lab, seed)
        if c["kind"] == "serve":
            self.server = fx.Server(self.graph, slots=c["slots"])

    def __del__(self):
        if self.server is not None:
            self.server.stop()
        if self.graph is not None:
            self.graph.close()


def prepare(case, seed):
    return State(case, seed)


# ---------------------------------------------------------------- one pass

def _columns(results):
    return {k: np.array([r[k] for r in results], np.int64) for k in FIELDS}


def _mined(graph, c):
    """The frequent set, one row a pattern, in a table with room for most graphs of the case (the
    set's size depends on the seed), and the candidates and frequent patterns of every level."""
    arr, levels = graph.mine_arrays(c["sigma"], c["lam"], c["edges"])
    n, rows = arr["n"].size, c["rows"]
    while rows < n:
        rows *= 2
    table = np.full((rows, 21), -1, np.int32)
    at = 0
    for k, width in (("n", 1), ("code_labels", 8), ("code_bits", 1), ("labels", 8), ("tau", 1), ("mis", 1), ("mni", 1)):
        a = arr[k].reshape(n, width)
        table[:n, at:at + width] = a.view(np.int32) if a.dtype.itemsize == 4 else a
        at += width
    return {"patterns": table, "levels": np.array([levels.get(k, (0, 0)) for k in range(2, 9)], np.int64)}


def run(s):
    c, g = s.case, s.graph
    kind = c["kind"]
    if kind == "query":
        return _columns([g.support(p[0], p[1], c["sigma"], c["lam"], mode=s.mode,
                                   edge_labels=p[2] if len(p) > 2 else None) for p in s.patterns])
    if kind == "batch":
        return _columns(g.support_batch(s.patterns, c["sigma"], c["lam"], s.mode))
    if kind == "mine":
        return _mined(g, c)
    if kind == "load":
        lab, src, dst, el = s.arrays
        g = fx.Graph(lab, src, dst, edge_labels=el, **s.options)
        out = _mined(g, c)
        info = g.info()
        g.close()
        out["info"] = np.array([info[k] for k in ("n_vertices", "n_arcs", "n_self_loops", "n_duplicates", "n_labels",
                                                  "max_degree")], np.int64)
        return out
    for i, p in enumerate(s.patterns):
        rc = s.server.submit(i, p[0], p[1], c["sigma"] * (1, 5, 20)[i % 3], (0.0, 0.5, 1.0)[i // 3 % 3], s.mode)
        if rc != fx.FLEXIS_OK:
            raise fx.FlexisError(rc, "submit")
    got = {}
    while len(got) < len(s.patterns):
        for rid, r, _ in s.server.poll():
            got[rid] = r
        time.sleep(1e-4)
    return _columns([got[i] for i in range(len(s.patterns))])


def work(case):
    """Bytes: the vertex labels and both directions of every edge read once (a load: the edge list
    read, the adjacency written), the patterns read and their results written.  No arithmetic but
    comparisons: a traversed arc counts as one operation."""
    arcs = case["ne"] * (1 if case.get("directed") else 2)
    per_pattern = 8 * 4 + 28 * 8 + fx.RESULT_DTYPE.itemsize
    n = case.get("count", 0)
    if case["kind"] == "load":
        return {"bytes": 4 * case["nv"] + 8 * case["ne"] + 4 * arcs + 4 * case["nv"], "flops": arcs}
    return {"bytes": 4 * case["nv"] + 4 * arcs + per_pattern * n, "flops": arcs}


# ---------------------------------------------------------------- plain values

def _mix(seed, v):
    """One SplitMix64 step from state seed XOR v."""
    m = (1 << 64) - 1
    z = ((seed ^ v) + 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


def _canonical(lab, edges):
    """The pattern relabelled to the order with the smallest (labels, not-adjacent bits by column)."""
    n = len(lab)
    adj = {(a, b) for a, b in edges} | {(b, a) for a, b in edges}
    best = min(itertools.permutations(range(n)),
               key=lambda p: ([lab[v] for v in p], [(p[i], p[j]) not in adj for j in range(n) for i in range(j)]))
    return [lab[v] for v in best], [{j for j in range(n) if (best[i], best[j]) in adj} for i in range(n)]


def _first_map(nbr, lab, pl, pa, order, root, used):
    """The lexicographically first map (by `order`) with order[0] at root and no used vertex."""
    bound = {order[0]: root}

    def rec(i):
        if i == len(order):
            return True
        u = order[i]
        back = [bound[w] for w in pa[u] if w in bound]
        for c in sorted(set.intersection(*(nbr[b] for b in back))):
            if lab[c] == pl[u] and c not in used and c not in bound.values():
                bound[u] = c
                if rec(i + 1):
                    return True
                del bound[u]
        return False

    return dict(bound) if lab[root] == pl[order[0]] and root not in used and rec(1) else None


def _order(pa, first):
    order = [first]
    while len(order) < len(pa):
        order.append(min(v for v in range(len(pa)) if v not in order and pa[v] & set(order)))
    return order


def exact(case, seed):
    """Queries on small undirected graphs: tau, mIS, MNI and the decision from the definitions."""
    if case["kind"] != "query" or case["nv"] > 4000 or case.get("directed") or case.get("edge_labels"):
        return None
    if case["ne"] > 8 * case["nv"] or case["count"] > 8:
        return None
    lab, src, dst, _ = make_graph(case, seed)
    nbr = [set() for _ in range(case["nv"])]
    for a, b in zip(src.tolist(), dst.tolist()):
        nbr[a].add(b)
        nbr[b].add(a)
    freq = np.bincount(lab)
    rank = {int(x): i for i, x in enumerate(sorted(np.flatnonzero(freq), key=lambda x: (freq[x], x)))}
    vl = [rank[int(x)] for x in lab]
    num = int(round(case["lam"] * 10**6))
    out = {k: [] for k in FIELDS}
    for pl, pe in make_patterns(case, lab, seed):
        n = len(pl)
        tau = case["sigma"] * ((n - 1) * num + 10**6) // (n * 10**6)
        need = max(tau, 1)
        cap = need if case["mode"] != "full" else None
        cl, pa = _canonical([rank[int(x)] for x in pl], pe.tolist())
        order = _order(pa, 0)
        used, mis = set(), 0
        for r in sorted((v for v in range(case["nv"]) if vl[v] == cl[0]), key=lambda v: (_mix(fx.DEFAULT_SEED, v), v)):
            m = _first_map(nbr, vl, cl, pa, order, r, used)
            if m:
                used |= set(m.values())
                mis += 1
                if mis == cap:
                    break
        mni = None
        if case["mode"] != "decide":
            mni = min(sum(1 for v in range(case["nv"]) if vl[v] == cl[u] and
                          _first_map(nbr, vl, cl, pa, _order(pa, u), v, ()) is not None) for u in range(n))
            mni = mni if cap is None else min(mni, cap)
        vals = dict(status=0, n=n, sigma=case["sigma"], tau=tau, cap=cap if cap is not None else -1, mis=mis,
                    mni=mni if mni is not None else -1, frequent=int(mis >= need), n_maps=0, mis_exact=-1)
        for k, v in vals.items():
            out[k].append(v)
    return {k: np.array(v, np.int64) if v else None for k, v in out.items()}
