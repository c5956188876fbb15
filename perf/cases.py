"""The isochrone queries whose time is measured, through the package's public
entry points: single queries on small and on country-sized road-like graphs,
ordinary batches, ragged ones, and full 64-lane batches, with every output the
library gives (isochrone edges, distances, vertices in range).

A case is a seeded grid graph (rows x cols, highway tiers "period:factor,..."),
a number of queries with limits drawn from [limit_lo, limit_hi], the call that
answers them and where its buffers live.  The graph, its hierarchy, the device
copy and the workspaces are what a user's program keeps and are made once per
process; a seed draws the queries (sources and limits)."""

import numpy as np
import torch

import paper_1512_09090_gb300 as P
from paper_1512_09090_gb300 import _lib, chcache, synth

# highway tiers of the repository's workloads: none, the 1000 x 1000 grid's, the 4243 x 4243 grid's
PLAIN, ONE_TIER, THREE_TIERS = "", "32:4", "16:2,128:4,1024:8"
LANDMARKS = 8       # as the benchmark adds them
FULL = 4243         # rows and columns of the full-size graph
CHAIN = 4           # batches of a chained pass, on two workspaces
LIST = 60000        # isochrone edges a program makes room for, per query
GRAPHS = {}         # (rows, cols, tiers) -> Graph


def case(rows, cols, tiers, queries, limit_lo, limit_hi, call, where="host", output="edges", limits="uniform"):
    return dict(rows=rows, cols=cols, tiers=tiers, queries=queries, limit_lo=limit_lo, limit_hi=limit_hi, call=call,
                where=where, output=output, limits=limits)


def listed():
    return [
        # the smallest call: one query on a town-sized graph (64 x 64, limit 1,500); launches and latency
        dict(case(64, 64, PLAIN, 1, 1500, 1500, "query"), name="town_k1"),
        # one interactive query on a city-region graph, the plain call with numpy arrays
        dict(case(1000, 1000, ONE_TIER, 1, 2000, 50000, "query"), name="region_k1"),
        # the allocation-free call of a latency-critical caller, at its largest batch
        dict(case(1000, 1000, ONE_TIER, 4, 2000, 50000, "noalloc", "device"), name="region_k4_noalloc"),
        # a small batch, the plain call
        dict(case(1000, 1000, ONE_TIER, 16, 2000, 50000, "query"), name="region_k16"),
        # a full batch whose caller also wants every distance (one-to-all, kept on the device)
        dict(case(1000, 1000, ONE_TIER, 64, 2000, 50000, "query", "device", "edges+dist"), name="region_k64_dist"),
        # ragged: odd sides, a partly filled batch, small limits mostly, vertices in range as well
        dict(case(1237, 811, ONE_TIER, 37, 600, 72000, "workspace", "device", "edges+range", "log"),
             name="ragged_k37_range"),
        # a state-sized graph, full batch, pinned host buffers
        dict(case(2000, 2000, THREE_TIERS, 64, 3600, 72000, "query", "pinned"), name="state_k64"),
        # one query with a small range on it, sweep restricted by landmark bounds
        dict(case(2000, 2000, THREE_TIERS, 1, 3600, 3600, "restricted", "device"), name="state_k1_restricted"),
        # the full-size graph, one query per launch
        dict(case(FULL, FULL, THREE_TIERS, 1, 3600, 72000, "workspace", "device"), name="full_k1"),
        # 16 sources with one shared limit
        dict(case(FULL, FULL, THREE_TIERS, 16, 36000, 36000, "workspace", "device"), name="full_k16"),
        # the headline end to end: 64 queries with uneven limits, pinned host buffers
        dict(case(FULL, FULL, THREE_TIERS, 64, 3600, 72000, "query", "pinned"), name="full_k64"),
        # the same as a server runs it: batches chained on two workspaces
        dict(case(FULL, FULL, THREE_TIERS, 64, 3600, 72000, "chained", "device"), name="full_k64_chained"),
    ]


def draw(rng):
    def logint(lo, hi):
        return min(hi, max(lo, round(lo * (hi / lo) ** rng.random())))

    queries = logint(1, 64)
    if rng.random() < 0.25:  # the full-size graph
        rows, cols, tiers = FULL, FULL, THREE_TIERS
    else:                    # from a town to a state, sides of their own (odd ones, oblong ones)
        rows, cols = logint(64, 1600), logint(64, 1600)
        tiers = rng.choice((PLAIN, ONE_TIER, THREE_TIERS))
    # limits from a few streets to most of the map (about 12 per row and column), 72,000 at most
    most = min(72000, 12 * (rows + cols))
    lo = logint(min(600, most // 4), most // 2)
    hi = logint(lo, most)
    call, where, output = rng.choice((("query", "host", "edges"), ("query", "pinned", "edges"),
                                      ("query", "device", "edges"), ("workspace", "device", "edges"),
                                      ("workspace", "device", "edges+range"), ("query", "device", "edges+dist"),
                                      ("restricted", "device", "edges"), ("noalloc", "device", "edges")))
    if call == "noalloc":
        queries = min(queries, 4)
    if rows * cols > (1 << 20) and (call in ("noalloc", "restricted") or output == "edges+dist"):
        call, output = "workspace", "edges"
    return case(rows, cols, tiers, queries, lo, hi, call, where, output, rng.choice(("uniform", "log")))


class Graph:
    """A road graph, its device copy, and the workspaces a program keeps on it."""

    def __init__(self, rows, cols, tiers):
        spec = dict(rows=rows, cols=cols, highways=tuple(tuple(int(x) for x in t.split(":"))
                                                         for t in tiers.split(",") if t), seed=1)
        named = [n for n, w in synth.WORKLOADS.items() if {**w, "seed": 1} == spec]
        if named:  # hierarchies of the repository's own workloads may lie in its cache
            try:
                self.road, self.ch = chcache.workload_graph_and_ch(named[0], log=lambda *a: None)
            except P.IsoError:
                named = []
        if not named:
            self.road = synth.grid_road_graph(**spec)
            self.ch = P.iso_build_ch(self.road.n, self.road.tail, self.road.head, self.road.weight)
        self.n = self.road.n
        self.starts = np.flatnonzero(np.bincount(self.road.tail, minlength=self.n) > 0)
        self.dev = P.iso_upload_graph(self.ch)
        self.kept = {}

    def workspaces(self, count, lanes, **opts):
        key = (count, lanes, tuple(sorted(opts.items())))
        if key not in self.kept:
            if opts.get("restrict_sweep") and not self.dev.landmarks:
                self.dev.add_landmarks(self.ch, LANDMARKS)
            self.kept[key] = [P.Workspace(self.dev, lanes, use_cuda_graph=1, **opts) for _ in range(count)]
        return self.kept[key]


def graph_of(c):
    key = (c["rows"], c["cols"], c["tiers"])
    if key not in GRAPHS:
        GRAPHS[key] = Graph(*key)
    return GRAPHS[key]


def batches_of(c):
    return CHAIN if c["call"] == "chained" else 1


def queries_of(c, seed):
    """Sources and limits of the case's batches, from the seed alone."""
    rng = np.random.default_rng(seed)
    starts, k = graph_of(c).starts, c["queries"]
    lo, hi = c["limit_lo"], c["limit_hi"]
    got = []
    for _ in range(batches_of(c)):
        src = starts[rng.integers(0, starts.size, size=k)].astype(np.int32)
        if c["limits"] == "log":
            tau = np.rint(np.exp(rng.uniform(np.log(lo), np.log(hi), size=k))).astype(np.int32)
        else:
            tau = rng.integers(lo, hi + 1, size=k).astype(np.int32)
        got.append((src, tau))
    return got


def prepare(c, seed):
    g = graph_of(c)
    s = dict(case=c, g=g, k=c["queries"], inputs=queries_of(c, seed))
    k, batches = c["queries"], batches_of(c)
    cap = LIST * k
    s["off"] = [np.zeros(k + 1, np.int64) for _ in range(batches)]
    s["arcs"] = [np.zeros(cap, np.int32) for _ in range(batches)]  # where the answers are kept
    if c["where"] == "pinned":
        s["inputs"] = [tuple(torch.from_numpy(x).pin_memory().numpy() for x in q) for q in s["inputs"]]
        s["off"] = [torch.zeros(k + 1, dtype=torch.int64).pin_memory().numpy() for _ in range(batches)]
        s["arcs"] = [torch.zeros(cap, dtype=torch.int32).pin_memory().numpy() for _ in range(batches)]
    elif c["where"] == "device":
        s["inputs"] = [tuple(torch.from_numpy(x).cuda() for x in q) for q in s["inputs"]]
        s["arcs"] = [torch.zeros(cap, dtype=torch.int32, device="cuda") for _ in range(batches)]
    if c["output"] == "edges+dist":
        s["dist"] = torch.zeros(k, g.n, dtype=torch.int32, device="cuda")
    if c["output"] == "edges+range":
        s["bits"] = torch.zeros(k, (g.n + 31) // 32, dtype=torch.int32, device="cuda")
    if c["call"] in ("workspace", "restricted"):
        s["ws"] = g.workspaces(1, k, **(dict(restrict_sweep=1) if c["call"] == "restricted" else {}))
    if c["call"] == "chained":
        s["ws"] = g.workspaces(2, k)
    return s


def run(s):
    c, g = s["case"], s["g"]
    src, tau = s["inputs"][0]
    off, arcs = s["off"][0], s["arcs"][0]
    if c["call"] == "query" and c["where"] == "host":
        # the plain call: numpy arrays in, new numpy arrays out, kept in the program's own
        off, got, _ = P.iso_query(g.dev, src, tau)
        arcs[:got.shape[0]] = got
        return [off, arcs]
    if c["call"] == "query":
        dist = s.get("dist")
        P.iso_query(g.dev, src, tau, out_offsets=off, out_arcs=arcs, out_dist=dist, use_cuda_graph=1)
        return [off, arcs] if dist is None else [off, arcs, dist]
    if c["call"] == "noalloc":
        _lib.iso_query_noalloc(g.dev, src, tau, off, arcs)
        return [off, arcs]
    if c["call"] == "chained":
        # batch b on workspace b % 2, each behind the sweep of the one before;
        # a workspace's batch is collected before its next one
        ws, prev, last = s["ws"], None, len(s["inputs"]) - 1
        for b in range(last + 3):
            if b >= 2:
                ws[b % 2].collect(out_offsets=s["off"][b - 2], out_arcs=s["arcs"][b - 2])
            if b <= last:
                ws[b % 2].submit(*s["inputs"][b], after=prev)
                prev = ws[b % 2]
        return [s["off"], s["arcs"]]
    w = s["ws"][0]
    w.submit(src, tau)
    w.collect(out_offsets=off, out_arcs=arcs)
    return [off, arcs, w.collect_range(s["bits"])] if c["output"] == "edges+range" else [off, arcs]


def work(c):
    """One pass over the downward arcs (8 bytes; about five per vertex on these
    grids) and the input arcs (head, 4 bytes; about 3.8 per vertex) with their
    offsets, an in-range bit per query and vertex written and read, about
    rows + cols isochrone edges per query written; distances and range bitsets
    where they are returned.  An add and a minimum per downward arc and query."""
    n, k, b = c["rows"] * c["cols"], c["queries"], batches_of(c)
    bytes_ = n * (5 * 8 + 3.8 * 4 + 8) + 2 * n * k / 8 + 4 * k * (c["rows"] + c["cols"])
    if c["output"] == "edges+dist":
        bytes_ += 4 * n * k
    if c["output"] == "edges+range":
        bytes_ += n * k / 8
    return {"bytes": b * bytes_, "flops": b * 2.0 * 5 * n * k}


def exact(c, seed):
    """Label-correcting distances in 64 bits over all input arcs, then the arcs
    with one endpoint in range; only where that is quick."""
    n, k = c["rows"] * c["cols"], c["queries"]
    if n * k > 4_000_000 or c["output"] != "edges" or c["call"] == "chained":
        return None
    road = graph_of(c).road
    tail, head, w = (torch.from_numpy(x.astype(np.int64)).cuda() for x in (road.tail, road.head, road.weight))
    (src, tau), far = queries_of(c, seed)[0], 1 << 40
    off, arcs = [0], []
    for s, t in zip(src.tolist(), tau.tolist()):
        d = torch.full((n,), far, dtype=torch.int64, device="cuda")
        d[s] = 0
        while True:
            via = d[tail] + w
            nd = d.scatter_reduce(0, head, torch.where(via <= t, via, far), "amin")
            if torch.equal(nd, d):
                break
            d = nd
        inside = d <= t
        arcs.append(torch.nonzero(inside[tail] != inside[head]).flatten().to(torch.int32).cpu().numpy())
        off.append(off[-1] + arcs[-1].size)
    kept = np.zeros(LIST * k, np.int32)
    kept[:off[-1]] = np.concatenate(arcs)
    return [np.array(off, np.int64), kept]
