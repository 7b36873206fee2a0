"""The work that users of this library have it do, as cases that a timer can run.

A case names an entry point ("api"), the graph it runs on and the query or
queries: listed() gives fixed ones, draw() others of the same ranges,
prepare() makes a case's inputs on the GPU from a seed, run() makes one pass
through the public Python API and returns what it computes.

Graphs (random from the seed; the shapes of the repository's own workloads):
  uniform   uniform endpoints and times, already in time order
  powerlaw  out-degrees of tail exponent 2.1, destinations by preferential
            attachment, times from a daily rhythm with 30% of the edges in
            bursts, 10% of the edges answered within an hour; unsorted
  hubs      both endpoints of tail exponent 1.8, a fifth of them on the top
            0.01% of the nodes, 16 edge labels, uniform times; unsorted
"""
import math
import random

import numpy as np
import torch

import paper_2310_02800_gb300 as tmg

DAY = 86_400
SECONDS_PER_EDGE = 9.4608      # 10M edges over three years: the power-law graphs' rate


def listed():
    return [
        # The smallest call: a small network's triangles, listed; launches and latency are all there is.
        {"name": "tiny_cycle3_rows", "api": "enumerate", "graph": "uniform", "nodes": 1_000, "edges": 20_000,
         "span": 1_000_000, "family": "cycle", "k": 3, "delta": 100_000, "cap": 65_536},
        # A real-time loop: a handful of standing queries re-counted on a small recent graph without allocating.
        {"name": "noalloc_8_queries_200k", "api": "count_noalloc", "graph": "powerlaw", "nodes": 20_000,
         "edges": 200_003, "span": 1_892_160, "queries": 8, "mix": 5, "delta": 3_600},
        # One shard of a large graph's roots (a rank's share, or a sample for a cost estimate), per-root counts.
        {"name": "shard_10m_cycle4_per_root", "api": "count_roots", "graph": "powerlaw", "nodes": 1_000_000,
         "edges": 10_000_000, "span": 94_608_000, "family": "cycle", "k": 4, "delta": 3_600, "parts": 61, "part": 30},
        # Motif features per edge of a mid-sized network: how many ping-pongs each edge starts.
        {"name": "count_1m_pingpong4_per_root", "api": "count", "graph": "powerlaw", "nodes": 100_000,
         "edges": 1_000_000, "span": 9_460_800, "family": "pingpong", "k": 4, "delta": 3_600, "per_root": True},
        # The benchmark step: four query shapes, each counted and its rows listed into capped buffers.
        {"name": "rows_batch_10m_4_queries", "api": "enumerate_batch", "graph": "powerlaw", "nodes": 1_000_000,
         "edges": 10_000_000, "span": 94_608_000, "queries": 4, "mix": -1, "delta": 3_600, "cap": 1 << 26},
        # Many standing queries of uneven size over the resident benchmark graph, counted in one launch.
        {"name": "count_batch_10m_64_queries", "api": "count_batch", "graph": "powerlaw", "nodes": 1_000_000,
         "edges": 10_000_000, "span": 94_608_000, "queries": 64, "mix": 2, "delta": 3_600},
        # Money flow over most of a day: long windows, a deep tree per root, one number back.
        {"name": "count_10m_path4_15h", "api": "count", "graph": "powerlaw", "nodes": 1_000_000, "edges": 10_000_000,
         "span": 94_608_000, "family": "path", "k": 4, "delta": 54_000, "per_root": False},
        # Edge-labelled paths with per-hop limits on a hub-skewed graph (odd sizes).
        {"name": "hubs_20m_path5_labels_gaps", "api": "count", "graph": "hubs", "nodes": 2_000_001,
         "edges": 20_000_003, "span": 30 * DAY, "family": "path", "k": 5, "delta": 7_200, "per_root": False,
         "edge_labels": True, "gap": 600},
        # The largest search: a dense rare motif (a 4-cycle, then both chords) on 100M hub-skewed edges.
        {"name": "hubs_100m_chorded_cycle", "api": "count", "graph": "hubs", "nodes": 10_000_000,
         "edges": 100_000_000, "span": 30 * DAY, "family": "chorded", "k": 6, "delta": 7_200, "per_root": False},
        # Constraints in earnest: 4-cycles with node labels, gaps and an anti-edge, each edge's share counted.
        {"name": "count_3m_cycle4_labels_gaps_anti", "api": "count", "graph": "powerlaw", "nodes": 300_000,
         "edges": 3_000_000, "span": 28_382_400, "family": "cycle", "k": 4, "delta": 3_600, "per_root": True,
         "node_labels": True, "gap": 1_800, "anti": True},
        # From host arrays to the answer and back out: load an unsorted edge list, list every match, map ids back.
        {"name": "load_1m_rows", "api": "load_rows", "graph": "powerlaw", "nodes": 100_000, "edges": 1_000_001,
         "span": 9_460_800, "family": "cycle", "k": 3, "delta": 3_600, "cap": 1 << 20},
        # A new day's graph: 10M unsorted edges in page-locked host arrays loaded, counted per edge and freed.
        {"name": "load_10m_count", "api": "load_count", "graph": "powerlaw", "nodes": 1_000_000, "edges": 10_000_000,
         "span": 94_608_000, "family": "cycle", "k": 3, "delta": 3_600, "per_root": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    api = rng.choice(["enumerate", "count_noalloc", "count_roots", "count", "count", "enumerate_batch", "count_batch",
                      "load_rows", "load_count", "hubs_labels", "hubs_chorded", "constraints"])
    if api.startswith("hubs"):
        edges = _log(rng, 2_000_000, 30_000_000)
        c = {"api": "count", "graph": "hubs", "nodes": edges // 10 + rng.randrange(7), "edges": edges,
             "span": 30 * DAY, "delta": _log(rng, 2_400, 7_200), "per_root": True}
        if api == "hubs_chorded":
            return dict(c, family="chorded", k=6)
        k = rng.randint(3, 5) if edges > 10_000_000 else rng.randint(3, 4)
        return dict(c, family="path", k=k, edge_labels=True, gap=_log(rng, 300, 1_200))
    if api in ("count_roots", "constraints"):
        edges = _log(rng, 1_000_000, 10_000_000)
    else:
        edges = _log(rng, 20_000, 10_000_000)
    c = {"api": api, "graph": "powerlaw", "nodes": edges // 10 + rng.randrange(9), "edges": edges,
         "span": int(edges * SECONDS_PER_EDGE * rng.uniform(0.8, 1.25))}
    if api in ("count_noalloc", "count_batch", "enumerate_batch"):
        most = 8 if api == "enumerate_batch" else 64
        c.update(queries=_log(rng, 2, most), mix=rng.randrange(1, 1000), delta=_log(rng, 600, 3_600))
        if api == "enumerate_batch":
            c["cap"] = _log(rng, 1_000, 10_000_000)
        return c
    if api == "constraints":
        delta = _log(rng, 1_800, 7_200)
        return dict(c, api="count", family="cycle", k=rng.randint(3, 4), delta=delta, per_root=True,
                    node_labels=rng.random() < 0.7, gap=delta // rng.randint(1, 3), anti=rng.random() < 0.7)
    family = rng.choice(["cycle", "path", "outstar", "instar", "pingpong"])
    k = rng.randint(*{"cycle": (3, 5), "path": (2, 5), "outstar": (2, 5), "instar": (2, 3), "pingpong": (2, 5)}[family])
    lo, hi = {"cycle": (1_800, 7_200), "path": (300, 7_200), "outstar": (120, 3_600), "instar": (60, 1_800),
              "pingpong": (1_800, DAY)}[family]
    c.update(family=family, k=k, delta=_log(rng, lo, hi))
    if api in ("enumerate", "load_rows"):
        c["cap"] = _log(rng, 100, 1_000_000)
    elif api == "count_roots":
        c["parts"] = rng.randint(2, 64)
        c["part"] = rng.randrange(c["parts"])
    else:
        c["per_root"] = family in ("cycle", "pingpong")
    return c


# ------------------------------------------------------------------ queries

FAMILIES = {
    "cycle": lambda k: [(i, (i + 1) % k) for i in range(k)],
    "path": lambda k: [(i, i + 1) for i in range(k)],
    "outstar": lambda k: [(0, i) for i in range(1, k + 1)],
    "instar": lambda k: [(i, 0) for i in range(1, k + 1)],
    "pingpong": lambda k: [(i % 2, 1 - i % 2) for i in range(k)],
    "chorded": lambda k: [(0, 1), (1, 2), (2, 3), (3, 0), (0, 2), (1, 3)],
}


def _motif(case):
    edges = FAMILIES[case["family"]](case["k"])
    delta, n = case["delta"], 1 + max(max(e) for e in edges)
    fixed = random.Random(3)       # the query's own constants: one program's query, whatever the graph
    return tmg.make_motif(
        edges, delta,
        gaps=[case["gap"]] * (len(edges) - 1) if case.get("gap") else None,
        elabel=[fixed.randrange(16) for _ in edges] if case.get("edge_labels") else None,
        nlabel=[fixed.randrange(2) for _ in range(n)] if case.get("node_labels") else None,
        anti=[(1, 0, 0, delta // 4)] if case.get("anti") else None)


def _motifs(case):
    """The queries of a batch: the benchmark's four (mix -1), or a seeded mix of shapes and windows."""
    if case["mix"] < 0:
        four = [("cycle", 3), ("cycle", 4), ("outstar", 3), ("pingpong", 4)]
        return [tmg.make_motif(FAMILIES[f](k), case["delta"]) for f, k in four]
    rng = random.Random(case["mix"])
    got = []
    for _ in range(case["queries"]):
        family, k = rng.choice(["cycle", "outstar", "path", "pingpong"]), rng.randint(2, 6)
        if family == "outstar":
            k = min(k, 5)
        if family == "cycle" and k == 2:
            family = "pingpong"
        got.append(tmg.make_motif(FAMILIES[family](k), _log(rng, 60, case["delta"])))
    return got


# ------------------------------------------------------------------- graphs

def _uniform(n, m, span, gen):
    dev = gen.device
    src = torch.randint(0, n, (m,), device=dev, generator=gen)
    dst = torch.randint(0, n - 1, (m,), device=dev, generator=gen)
    dst += dst >= src
    t = torch.randint(0, span, (m,), device=dev, generator=gen).sort().values
    return src.int(), dst.int(), t


def _ranks(n, m, alpha, first, gen):
    """m node ranks in [first, n) of weights (rank + 1)^(-1 / (alpha - 1))."""
    om = 1.0 - 1.0 / (alpha - 1.0)
    lo, hi = (first + 1.0) ** om, (n + 1.0) ** om
    u = torch.rand(m, device=gen.device, generator=gen, dtype=torch.float64)
    return (u.mul_(hi - lo).add_(lo).pow_(1.0 / om) - 1.0).long().clamp_(first, n - 1)


def _no_loops(src, dst, n, gen):
    other = torch.randint(0, n - 1, src.shape, device=gen.device, generator=gen)
    other += other >= src
    return torch.where(src == dst, other, dst)


def _daily(u, span):
    """Times in [0, span) of a daily rhythm of amplitude 0.8, from uniform draws u."""
    w, amp = 2.0 * math.pi / DAY, 0.8
    s = u * (span + amp / w * (1.0 - math.cos(w * span)))
    t = s.clone()
    for _ in range(16):
        t -= (t + amp / w * (1.0 - torch.cos(w * t)) - s) / (1.0 + amp * torch.sin(w * t))
        t = torch.minimum(torch.maximum(t, s - 2.0 * amp / w), s)
    return t.clamp_(0.0, span - 1.0)


def _powerlaw(n, m, span, gen):
    dev = gen.device

    def rand(k):
        return torch.rand(k, device=dev, generator=gen, dtype=torch.float64)

    base = max(1, int(m / 1.1))
    src = torch.randperm(n, device=dev, generator=gen)[_ranks(n, base, 2.1, 0, gen)]
    # destinations: copy that of a random earlier edge with probability 1 / 1.1, else uniform
    at = torch.arange(base, device=dev)
    earlier = (rand(base) * at).long()
    copied = rand(base) < 1.0 / 1.1
    copied[0] = False
    todo = copied.nonzero().squeeze(1)
    while todo.numel():
        at[todo] = earlier[at[todo]]
        todo = todo[copied[at[todo]]]
    dst = torch.randint(0, n, (base,), device=dev, generator=gen)[at]
    dst = _no_loops(src, dst, n, gen)
    bursts = int(base * 0.3 / 50.0) + 1
    centre = _daily(rand(bursts), span)[torch.randint(0, bursts, (base,), device=dev, generator=gen)]
    in_burst = (centre - 300.0 * torch.log1p(-rand(base))).clamp_(max=span - 1.0)
    t = torch.where(rand(base) < 0.3, in_burst, _daily(rand(base), span)).long()
    back = torch.randperm(base, device=dev, generator=gen)[: m - base]      # answered within an hour
    t_back = t[back] + 1 + torch.randint(0, 3_600, back.shape, device=dev, generator=gen)
    return torch.cat([src, dst[back]]).int(), torch.cat([dst, src[back]]).int(), torch.cat([t, t_back])


def _hubs(n, m, span, gen):
    dev = gen.device
    hubs = max(1, n // 10_000)
    node = torch.randperm(n, device=dev, generator=gen)

    def ends():
        rank = _ranks(n, m, 1.8, hubs, gen)
        hub = torch.randint(0, hubs, (m,), device=dev, generator=gen)
        return node[torch.where(torch.rand(m, device=dev, generator=gen) < 0.2, hub, rank)]

    src = ends()
    dst = _no_loops(src, ends(), n, gen)
    t = torch.randint(0, span, (m,), device=dev, generator=gen)
    return src.int(), dst.int(), t


def _edges(case, seed):
    """(src, dst, t, edge labels, node labels) of the case's graph, on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    make = {"uniform": _uniform, "powerlaw": _powerlaw, "hubs": _hubs}[case["graph"]]
    n, m = case["nodes"], case["edges"]
    src, dst, t = make(n, m, case["span"], gen)
    elabel = nlabel = None
    if case["graph"] == "hubs":
        elabel = torch.randint(0, 16, (m,), device="cuda", generator=gen, dtype=torch.uint8)
    if case.get("node_labels"):
        nlabel = torch.randint(0, 2, (n,), device="cuda", generator=gen, dtype=torch.uint8)
    return src, dst, t, elabel, nlabel


# --------------------------------------------------------------------- runs

def _page_locked(x):
    """A host copy of x as a numpy array in page-locked memory (the array keeps the tensor)."""
    return torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x).numpy()


def _row_buffer(cap, k):
    """A match buffer: rows past the ones written stay -1, so that all of it is an output."""
    return torch.full((cap, k), -1, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    api = case["api"]
    src, dst, t, elabel, nlabel = _edges(case, seed)
    if api in ("load_rows", "load_count"):
        host = _page_locked if api == "load_count" else (lambda x: x.cpu().numpy())
        s = {"case": case, "src": host(src), "dst": host(dst), "t": host(t), "motif": _motif(case)}
        if api == "load_rows":
            s["rows"] = _row_buffer(case["cap"], case["k"])
        elif case["per_root"]:
            s["per_root"] = torch.zeros(case["edges"], dtype=torch.int64, device="cuda")
        return s
    g = tmg.Graph.load(case["nodes"], src, dst, t, elabel, nlabel)
    s = {"case": case, "graph": g}
    if "queries" in case:
        s["queries"] = [g.compile(m) for m in _motifs(case)]
    else:
        s["query"] = g.compile(_motif(case))
    if api == "enumerate":
        s["rows"] = _row_buffer(case["cap"], case["k"])
    elif api == "enumerate_batch":
        s["rows"] = [_row_buffer(case["cap"], q.k) for q in s["queries"]]
    elif api == "count_noalloc":
        s["totals"] = torch.zeros(case["queries"], dtype=torch.int64, device="cuda")
    elif api == "count_roots":
        m, parts = case["edges"], case["parts"]
        s["range"] = (m * case["part"] // parts, m * (case["part"] + 1) // parts)
        s["per_root"] = torch.zeros(s["range"][1] - s["range"][0], dtype=torch.int64, device="cuda")
    elif api == "count" and case["per_root"]:
        s["per_root"] = torch.zeros(case["edges"], dtype=torch.int64, device="cuda")
    return s


def run(state):
    api = state["case"]["api"]
    if api == "count":
        per_root = state.get("per_root")
        total = state["query"].count(per_root=per_root)
        return {"total": total} if per_root is None else {"total": total, "per_root": per_root}
    if api == "count_roots":
        total = state["query"].count_roots(*state["range"], per_root=state["per_root"])
        return {"total": total, "per_root": state["per_root"]}
    if api == "enumerate":
        written, total, truncated = state["query"].enumerate(state["rows"])
        return {"rows": state["rows"], "written": written, "total": total, "truncated": truncated}
    if api == "enumerate_batch":
        written, totals, truncated = state["graph"].enumerate_batch(state["queries"], state["rows"])
        return {"rows": state["rows"], "written": np.array(written), "totals": np.array(totals),
                "truncated": truncated}
    if api == "count_batch":
        return {"totals": np.array(state["graph"].count_batch(state["queries"]))}
    if api == "count_noalloc":
        return {"totals": state["graph"].count_batch_noalloc(state["queries"], state["totals"])}
    case = state["case"]
    g = tmg.Graph.load(case["nodes"], state["src"], state["dst"], state["t"])
    q = g.compile(state["motif"])
    if api == "load_count":
        per_root = state.get("per_root")
        total = q.count(per_root=per_root)
        got = {"total": total} if per_root is None else {"total": total, "per_root": per_root}
    else:
        written, total, _ = q.enumerate(state["rows"])
        got = {"total": total, "written": written, "rows": state["rows"], "edge_perm": g.edge_perm()}
    q.free()
    g.free()
    return got


def exact(case, seed):
    """Every output is whole numbers, which stay equal: no floating value to hold against 64 bits."""
    return None


def work(case):
    """A search reads each edge once (two ids and a time, labels where the query asks for them) and writes what
    is asked for per root; rows are left out, since their number is not known before the call.  A load reads the
    edge list and writes it in time order with its permutation and the two adjacency lists (time, neighbour and
    edge id per entry, offsets per node)."""
    m, n, api = case["edges"], case["nodes"], case["api"]
    if api == "count_roots":
        m = m // case["parts"]
    read = 16 * m + (m if case.get("edge_labels") else 0) + (n if case.get("node_labels") else 0)
    out = 8 * m if api == "count_roots" or case.get("per_root") else 0
    if api in ("load_rows", "load_count"):
        out += 16 * m + 20 * m + 32 * m + 8 * n + (8 * m if api == "load_rows" else 0)
    return {"bytes": read + out, "flops": 0}
