"""Performance cases: what a user of the library has it do, each through the public entry points.

A case is a dict of plain values.  Point sets and query radii follow the shapes of
workloads.py (uniform, mixed and clustered Gaussian points, road-like lines, the paper's
Normal and Skewed distributions, 3-D mixtures; fixed radii, or radii matched to the local
density so that the expected hit count is log-uniform), drawn on the GPU from the seed.
Every output is a whole number (ids, offsets, keys, coordinates), so two runs on the same
inputs give the same values.

  what     query   sfc_query_count on a built index, the total read back (a program grows its
                   result buffer by it), sfc_query_write
           step    sfc_rebuild over new points, then sfc_query_batch into kept buffers
           graph   the same step captured once as a CUDA graph, one launch per pass
           build   sfc_rebuild alone
           update  sfc_update: one batch of deletes and inserts on a built index
           host    sfc_query_batch_host: queries and results in page-locked host memory
           sort    sfc_sort_pairs on 60-bit keys
"""
import math

import numpy as np
import torch

import paper_2508_19891_gb300 as sfc

SIDE = 1 << 30
SIDE3 = 1 << 21


def _case(name, what, points, n, m=0, **more):
    c = {"name": name, "what": what, "points": points, "n": n, "m": m, "curve": "z", "cover": 0, "bounds": "binary",
         "norm": "disc", "radius": "matched", "k": 2000}
    c.update(more)
    return c


def listed():
    return [
        # one lookup against a resident index: an interactive "what is near here"
        _case("lookup-1", "query", "uniform", 1_000_003, 1, radius="fixed", k=20),
        # a few thousand lookups with tuned cover, the request batch of a service
        _case("requests-3e3", "query", "mixed", 2_000_003, 3001, cover=1, k=500),
        # the small workload of the tests and the benchmark as one simulation frame: points move,
        # the index is rebuilt and every 10th point asks for its neighbours, replayed as a graph
        _case("uniform-1e5-graph", "graph", "box20", 100_000, 10_000, radius="fixed", k=20),
        # the paper's Skewed points with square windows, odd sizes, default options
        _case("skewed-3e5-square", "step", "skewed", 300_007, 50_021, norm="square", radius="fixed", k=60),
        # the paper's Normal points with uniformly placed square windows (many nearly empty)
        _case("normal-1e7-square", "query", "normal", 10_000_000, 1_000_000, norm="square", radius="fixed", k=10),
        # the mixed workload at its ordinary size: queries at data points, 1 to 2,000 hits each
        _case("mixed-1e7", "query", "mixed", 10_000_000, 1_000_000, cover=1),
        # a few analyst's windows that each report hundreds of thousands of points
        _case("windows-2e5", "query", "uniform", 10_000_000, 129, radius="fixed", k=200_000),
        # the same index behind a host-buffer service: copies in and out are part of the call
        _case("host-1e5", "host", "mixed", 10_000_000, 100_003, cover=1, k=500),
        # road-like points on the Hilbert curve: rebuild and query, fixed radius of 25 spacings
        _case("roads-3e7-hilbert", "step", "roads", 30_000_000, 2_000_000, curve="h", radius="roads", k=50),
        # the dynamic workload: half a million points of a clustered set leave, as many arrive
        _case("update-5e7", "update", "clustered", 50_000_000, 500_000),
        # 3-D points: rebuild and balls at data points
        _case("mixed3d-1e7", "step", "mixed3", 10_000_000, 1_000_000, cover=1),
        # the benchmark's headline step: rebuild, model fit and 10^7 queries over 10^8 points
        _case("mixed-1e8-learned", "step", "mixed", 100_000_000, 10_000_000, cover=1, bounds="learned"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    what = rng.choice(["query", "query", "step", "step", "graph", "build", "update", "host", "sort"])
    points = rng.choice(["uniform", "mixed", "clustered", "normal", "skewed", "roads", "mixed3"])
    n = _log_int(rng, 10_000, 60_000_000)
    if what in ("update", "sort") and points == "mixed3":
        points = "clustered"
    if what == "sort":
        points = "keys"
    if what == "graph":
        n = min(n, 3_000_000)
    m = {"build": 0, "sort": 0, "update": _log_int(rng, 1, max(2, n // 20))}.get(what, _log_int(rng, 1, max(2, n // 10)))
    radius = "roads" if points == "roads" else ("matched" if points in ("mixed", "clustered", "mixed3") else "fixed")
    k = _log_int(rng, 4, min(2000, n // 20))
    # no more results than the largest listed case reports: up to 10^9 ids, 10^8 over the host link
    m = min(m, max(1, (100_000_000 if what == "host" else 1_000_000_000) // k)) if what != "update" else m
    return {"what": what, "points": points, "n": n, "m": m,
            "curve": "z" if points == "mixed3" else rng.choice(["z", "z", "h"]),
            "cover": rng.choice([0, 1]) if points == "mixed3" else rng.choice([0, 1, 1, 2]),
            "bounds": "binary" if points == "mixed3" or what == "update" else rng.choice(["binary", "learned"]),
            "norm": "disc" if points in ("mixed3", "mixed", "clustered", "roads") else rng.choice(["disc", "square"]),
            "radius": radius, "k": k}


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1_000_003 + 17)
    return g


def _clamp(xy, side):
    return xy.round_().clamp_(0, side - 1).to(torch.int32)


def _gauss_mix(g, n, n_uniform, dim, side, sigma, clusters):
    """Points, the squared distance to the own cluster's centre (inf for background points)."""
    centres = torch.rand((clusters, dim), generator=g, device="cuda", dtype=torch.float64) * side
    which = torch.randint(0, clusters, (n,), generator=g, device="cuda")
    xy = torch.randn((n, dim), generator=g, device="cuda", dtype=torch.float32).double().mul_(sigma).add_(centres[which])
    pts = _clamp(xy, side)
    r2 = (pts.double() - centres[which]).square_().sum(1)
    bg = torch.randint(0, n, (n,), generator=g, device="cuda") < n_uniform
    flat = torch.randint(0, side, (n, dim), generator=g, device="cuda", dtype=torch.int32)
    pts = torch.where(bg[:, None], flat, pts)
    return pts.contiguous(), r2.masked_fill_(bg, math.inf)


def _road_spacing(n):
    # 200,000 lines of about 30 segments of mean length 2^14 e^0.5, at n = 3 * 10^7 points
    return max(1, int(5400 * (30_000_000 / n) ** 0.5))


def _points(case, g):
    """int32 points and, for mixtures, each point's squared distance to its cluster's centre."""
    kind, n = case["points"], case["n"]
    clusters = max(1, min(1000, int(round(1000 * math.sqrt(n / 1e7)))))
    if kind == "uniform":
        return torch.randint(0, SIDE, (n, 2), generator=g, device="cuda", dtype=torch.int32), None
    if kind == "box20":
        return torch.randint(0, 1 << 20, (n, 2), generator=g, device="cuda", dtype=torch.int32), None
    if kind == "mixed":
        return _gauss_mix(g, n, n // 2, 2, SIDE, 2.0 ** 18, clusters)
    if kind == "clustered":
        return _gauss_mix(g, n, 0, 2, SIDE, 2.0 ** 18, clusters)
    if kind == "mixed3":
        return _gauss_mix(g, n, n // 2, 3, SIDE3, 2.0 ** 11, clusters)
    if kind == "normal":
        xy = torch.randn((n, 2), generator=g, device="cuda", dtype=torch.float32).double()
        return _clamp(xy.mul_(SIDE / 8).add_(SIDE / 2), SIDE), None
    if kind == "skewed":
        x = torch.randint(0, SIDE, (n,), generator=g, device="cuda").double()
        y = torch.rand((n,), generator=g, device="cuda", dtype=torch.float64).neg_().log1p_().mul_(-SIDE / 5).floor_()
        return _clamp(torch.stack([x, y], 1), SIDE), None
    # roads: lines of 150 points at jittered spacing, the heading a random walk that turns about
    # every eighth point (whole-number sums, the same on every run)
    per = 150
    lines = (n + per - 1) // per
    h = _road_spacing(n)
    head = torch.randint(0, 4096, (lines, 1), generator=g, device="cuda")
    turn = (torch.randn((lines, per), generator=g, device="cuda") * 230).to(torch.int64)
    turn *= (torch.randint(0, 8, (lines, per), generator=g, device="cuda") == 0)
    ang = (head + turn.cumsum(1)).double() * (2 * math.pi / 4096)
    step = h + torch.randint(-(h // 4) - 1, h // 4 + 1, (lines, per), generator=g, device="cuda").double()
    xy = torch.stack([(step * ang.cos()).round_().to(torch.int64), (step * ang.sin()).round_().to(torch.int64)], 2).cumsum(1)
    xy = xy + torch.randint(0, SIDE, (lines, 1, 2), generator=g, device="cuda")
    xy = xy.view(-1, 2)[:n].clamp_(0, SIDE - 1).to(torch.int32)
    return xy[torch.randperm(n, generator=g, device="cuda")].contiguous(), None


def _queries(case, g, pts, r2):
    """Centres and radii: at data points for matched and road radii, else uniform in the box."""
    n, m, k = case["n"], case["m"], case["k"]
    dim = pts.shape[1]
    side = {"box20": 1 << 20, "mixed3": SIDE3}.get(case["points"], SIDE)
    if case["radius"] == "fixed":
        q = torch.randint(0, side, (m, dim), generator=g, device="cuda", dtype=torch.int32)
        area = k * float(side) ** 2 / n
        d = math.sqrt(area) / 2 if case["norm"] == "square" else math.sqrt(area / math.pi)
        return q, torch.full((m,), max(1, int(round(d))), dtype=torch.int32, device="cuda")
    at = torch.randint(0, n, (m,), generator=g, device="cuda")
    q = pts[at].contiguous()
    if case["radius"] == "roads":
        return q, torch.full((m,), int(k / 2 * _road_spacing(n)), dtype=torch.int32, device="cuda")
    clusters = max(1, min(1000, int(round(1000 * math.sqrt(n / 1e7)))))
    n_u = 0 if case["points"] == "clustered" else n // 2
    sigma = 2.0 ** 11 if dim == 3 else 2.0 ** 18
    near = torch.exp(r2[at] / (-2 * sigma * sigma)) * ((n - n_u) / clusters / (math.sqrt(2 * math.pi) * sigma) ** dim)
    rho = near + n_u / float(side) ** dim + 1e-30
    kk = torch.exp(torch.rand((m,), generator=g, device="cuda", dtype=torch.float64) * math.log(k))
    d = (kk / (math.pi * rho)).sqrt() if dim == 2 else (kk / (4 / 3 * math.pi * rho)) ** (1 / 3)
    # a point far out in a cluster's tail has next to no density: its radius stays within 2 sigma
    # where there is no background, so that no query takes in whole clusters
    d = d.clamp(max=2 * sigma if n_u == 0 else side // 2)
    return q, d.round_().clamp_(1, side).to(torch.int32)


def _mean_hits(case):
    """Expected hits of a query: log-uniform radii give (k - 1) / ln k; a road's disc takes in
    about 6e-4 k^2 points of other lines."""
    k = case["k"]
    if case["radius"] == "matched":
        return (k - 1) / math.log(k)
    return k + (6e-4 * k * k if case["radius"] == "roads" else 0)


def _capacity(case):
    """Ids that a result buffer holds: two to three times the expected total (radii matched to
    the background density also reach into clusters), and room for a few queries in the densest
    parts when there are only a few."""
    n, m = case["n"], case["m"]
    few = min(m, 64) * (20 * case["k"] + (n // 200 if case["points"] in ("mixed", "clustered", "mixed3") else 0))
    return int(min(m * n, m * _mean_hits(case) * (2 if n > 30_000_000 else 3) + few))


def _options(case):
    o = {"cover_refine": case["cover"]}
    if case["points"] != "mixed3":
        o.update(bounds=case["bounds"], query_norm=case["norm"])
    return o


def _build(case, pts):
    if pts.shape[1] == 3:
        return sfc.sfc_build3(pts, **_options(case))
    return sfc.sfc_build(pts, case["curve"], **_options(case))


def prepare(case, seed):
    g = _gen(seed)
    if case["what"] == "sort":
        keys = torch.randint(0, 1 << 60, (case["n"],), generator=g, device="cuda", dtype=torch.int64)
        return {"what": "sort", "keys": keys}
    pts, r2 = _points(case, g)
    s = {"what": case["what"], "pts": pts, "index": _build(case, pts)}
    if case["what"] == "build":
        return s
    if case["what"] == "update":
        ins, _ = _points(dict(case, n=case["m"]), g)
        gone = torch.randperm(case["n"], generator=g, device="cuda")[:case["m"]].to(torch.int32)
        return dict(s, pts=None, ins=ins, gone=gone)
    q, d = _queries(case, g, pts, r2)
    s.update(q=q, d=d)
    # result buffers that a program keeps; ids beyond the total stay zero
    cap = _capacity(case)
    if case["what"] == "host":
        pin = {"q": q.cpu(), "d": d.cpu(), "off": torch.zeros(case["m"] + 1, dtype=torch.int64),
               "ids": torch.zeros(cap, dtype=torch.int32)}
        pin = {k: v.pin_memory() for k, v in pin.items()}
        return {"what": "host", "index": s["index"], "keep": pin, "cap": cap, "q": pin["q"].numpy(), "d": pin["d"].numpy(),
                "off": pin["off"].numpy().view(np.uint64), "ids": pin["ids"].numpy().view(np.uint32)}
    s.update(off=torch.zeros(case["m"] + 1, dtype=torch.int64, device="cuda"),
             ids=torch.zeros(cap, dtype=torch.int32, device="cuda"))
    if case["what"] == "graph":
        s["graph"] = sfc.sfc_graph_capture(s["index"], pts, q, d, s["off"], s["ids"])
    return dict(s, pts=None) if case["what"] == "query" else s


# ------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------

def run(state):
    what = state["what"]
    if what == "sort":
        return sfc.sfc_sort_pairs(state["keys"])
    index = state["index"]
    if what == "query":
        off = sfc.sfc_query_count(index, state["q"], state["d"], state["off"])
        total = int(off[-1].item())
        if total > state["ids"].numel():
            state["ids"] = torch.zeros(total, dtype=torch.int32, device="cuda")
        return off, sfc.sfc_query_write(index, state["q"], state["d"], off, state["ids"])
    if what == "host":
        sfc.sfc_query_batch_host(index, state["q"], state["d"], state["cap"], state["off"], state["ids"])
        return state["off"].view(np.int64), state["ids"].view(np.int32)
    if what == "update":
        # the points that arrived with this batch leave with the next one
        first = sfc.sfc_update(index, state["ins"], state["gone"])
        state["gone"] = torch.arange(first, first + state["ins"].shape[0], dtype=torch.int32, device="cuda")
        return sfc.sfc_get_sorted(index, copy=False)
    if what == "graph":
        state["graph"].launch()
        return state["off"], state["ids"]
    sfc.sfc_rebuild(index, state["pts"])
    if what == "build":
        return sfc.sfc_get_sorted(index, copy=False)
    return sfc.sfc_query_batch(index, state["q"], state["d"], state["off"], state["ids"])


def work(case):
    """Bytes and integer operations of one pass: each input read and each output written once.
    A query reads a point (8 bytes, 16 in 3-D) and an id for each hit at least, but no more than
    the arrays once, and writes 4 bytes for each."""
    n, m = case["n"], case["m"]
    dim = 3 if case["points"] == "mixed3" else 2
    if case["what"] == "sort":
        return {"bytes": 8 * n + 12 * n, "flops": 0}
    build = 4 * dim * n + 12 * n + (16 if dim == 3 else 8) * n   # points in; keys, ids and coordinates out
    if case["what"] == "build":
        return {"bytes": build, "flops": 0}
    if case["what"] == "update":
        return {"bytes": 2 * 20 * n + (8 + 4) * m, "flops": 0}
    hits = m * _mean_hits(case)
    seen = min(hits, n) * ((16 if dim == 3 else 8) + 4)
    query = m * (4 * dim + 4 + 8) + seen + 4 * hits
    rebuild = case["what"] in ("step", "graph")
    return {"bytes": int(query + (build if rebuild else 0)), "flops": int(hits * (2 * dim + dim))}
