"""Timed cases of the R-tree library: the work its users have it do.

Every case goes through the public Python entry points (``RTree``,
``RTree.range_select``, ``RTree.join``, ``Plan``,
``rtree_range_select_host``) on synthetic data of the workloads in
``paper_2309_16913_gb300/datagen.py``, drawn on the GPU.  A result's length
depends on the data, and results of different inputs are to have the same
shape here: so a case's own values seed its rectangles and queries, and the
seed then mirrors and swaps the axes (exact in float32), renumbers the
rectangles and reorders the queries, which gives other trees and other answers
of the same length.  A case is a dict of plain values:

  kind     select   a batch of range queries on a tree that is kept
           plan     the same through a graph-captured plan that is kept
           host     the same with the result in page-locked host memory
           build    a tree built from new rectangles, then a batch on it
           join     the join of two trees that are kept
           layers   two trees built from new rectangles, then joined
  n, m     rectangles of the tree (of the second tree)
  q        queries of the batch
  data     uniform, or mixed (80% in 64 Gaussian clusters, 20% uniform)
  rows     shuffled (ids say nothing about the position) or tiled (rows stored
           region by region, so that nearby rectangles have nearby ids)
  queries  selective (squares, selectivity log-uniform in [sel_lo, sel_hi]),
           small (sides uniform in [0, 0.01]), windows (sides uniform in
           [0.05, 0.2]) or uneven (99% sides in [0, 1e-3], 1% windows)

All outputs are whole numbers (offsets, ids, pairs) that the float32
comparisons decide exactly, so there is nothing for a 64-bit reference to add.
"""
import json
import math
import zlib

import torch

from paper_2309_16913_gb300 import rtree as rt

SIDE_LO, SIDE_HI = 1e-5, 1e-3   # log-uniform sides of the mixed data
JOIN_SIDE = 5e-4                # uniform sides of the join's data, in [0, JOIN_SIDE]
PLAIN_SIDE = 1e-3               # uniform sides of the uniform data, in [0, PLAIN_SIDE]


def listed():
    return [
        # one lookup by a program that asks one question at a time: default options
        dict(name="single_query", kind="select", n=1_000_003, q=1, data="mixed", rows="shuffled",
             queries="selective", sel_lo=1e-5, sel_hi=1e-4, fanout=16, layout="soa", order="input",
             mapping="auto", unsorted=False),
        # a serving loop's batch: a few hundred waiting requests through a captured plan
        dict(name="plan_batch", kind="plan", n=10_000_000, q=200, data="mixed", rows="shuffled",
             queries="selective", sel_lo=1e-7, sel_hi=1e-3, fanout=64, layout="aos", mapping="auto"),
        # the plain workload with the library's default options
        dict(name="plain", kind="select", n=100_000, q=1000, data="uniform", rows="shuffled",
             queries="small", fanout=16, layout="soa", order="input", mapping="auto", unsorted=False),
        # a handful of map windows, each covering a large part of the data
        dict(name="windows", kind="select", n=10_000_000, q=48, data="mixed", rows="shuffled",
             queries="windows", fanout=64, layout="aos", order="input", mapping="auto", unsorted=False),
        # an ordinary batch with the default options on data stored region by region
        dict(name="tiled_default", kind="select", n=2_000_003, q=100_003, data="mixed", rows="tiled",
             queries="selective", sel_lo=1e-6, sel_hi=1e-3, fanout=16, layout="soa", order="input",
             mapping="auto", unsorted=False),
        # candidates for a later filter, which needs no order inside a query
        dict(name="unsorted", kind="select", n=3_000_017, q=200_000, data="mixed", rows="shuffled",
             queries="selective", sel_lo=1e-6, sel_hi=1e-3, fanout=32, layout="lohi", order="input",
             mapping="auto", unsorted=True),
        # the scaled workload's batch on its index (tuned options)
        dict(name="scaled", kind="select", n=10_000_000, q=1_000_000, data="mixed", rows="shuffled",
             queries="selective", sel_lo=1e-6, sel_hi=1e-3, fanout=64, layout="aos", order="hilbert",
             mapping="auto", unsorted=False),
        # the uneven workload: most queries tiny, one in a hundred a large window
        dict(name="uneven_plan", kind="plan", n=10_000_000, q=100_000, data="mixed", rows="shuffled",
             queries="uneven", fanout=64, layout="aos", mapping="auto"),
        # the result wanted in host memory
        dict(name="to_host", kind="host", n=10_000_000, q=30_011, data="mixed", rows="shuffled",
             queries="selective", sel_lo=1e-6, sel_hi=1e-3, fanout=128, layout="lohi", order="hilbert",
             mapping="auto", unsorted=False),
        # an index over data that moves: built anew, then asked a batch of queries
        dict(name="build", kind="build", n=10_000_000, q=1000, data="mixed", rows="shuffled",
             queries="selective", sel_lo=1e-6, sel_hi=1e-3, fanout=64, layout="aos", order="input",
             mapping="auto", unsorted=False),
        # the join workload on two kept trees
        dict(name="join", kind="join", n=2_000_000, m=2_000_000, fanout=32, layout="soa",
             sort_children=False, fanout_m=32),
        # two map layers of unlike size indexed and overlaid, with the sorted-node prunings
        dict(name="layers", kind="layers", n=150_001, m=400_009, fanout=16, layout="aos",
             sort_children=True, fanout_m=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    fanout = rng.choice((8, 16, 16, 32, 64, 64, 128))
    layout = rng.choice(("soa", "aos", "lohi"))
    kind = rng.choice(("select", "select", "select", "plan", "host", "build", "join", "layers"))
    if kind in ("join", "layers"):
        return dict(kind=kind, n=_log_int(rng, 5_000, 2_000_000), m=_log_int(rng, 5_000, 2_000_000),
                    fanout=max(16, fanout), layout=layout, sort_children=rng.random() < 0.5,
                    fanout_m=rng.choice((16, 32, 64)))
    n = _log_int(rng, 20_000, 10_000_000)
    c = dict(kind=kind, n=n, q=1, data=rng.choice(("mixed", "mixed", "uniform")),
             rows=rng.choice(("shuffled", "shuffled", "tiled")),
             queries=rng.choice(("selective", "selective", "selective", "small", "uneven", "windows")),
             fanout=fanout, layout=layout, mapping="auto")
    if c["queries"] == "selective":
        c["sel_lo"], c["sel_hi"] = rng.choice(((1e-6, 1e-3), (1e-7, 1e-4), (1e-5, 1e-2)))
    top = {"select": 1_000_000, "plan": 100_000, "host": 60_000, "build": 100_000}[kind]
    ids_top = {"select": 6e8, "plan": 1.5e8, "host": 4e7, "build": 1e8}[kind]
    top = int(max(1, min(top, ids_top / max(_hits_per_query(c), 1e-9))))
    c["q"] = _log_int(rng, 1, top)
    if kind != "plan":
        c["order"] = rng.choice(("input", "hilbert"))
        c["unsorted"] = kind == "select" and rng.random() < 0.2
    if not c.get("unsorted") and rng.random() < 0.15:
        c["mapping"] = "work_queue"  # its unsorted order is not fixed
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _case_seed(c):
    return zlib.crc32(json.dumps({k: v for k, v in c.items() if k != "name"}, sort_keys=True).encode())


def _perm(g, n):
    return torch.randperm(n, generator=g, device="cuda")


def _turn(g):
    """One of the square's eight symmetries, drawn from g: a function on [n, 4] boxes."""
    fx, fy, swap = (torch.rand(3, generator=g, device="cuda") < 0.5).tolist()

    def turn(b):
        x0, y0, x1, y1 = b.unbind(1)
        x0, x1 = (-x1, -x0) if fx else (x0, x1)
        y0, y1 = (-y1, -y0) if fy else (y0, y1)
        return torch.stack((y0, x0, y1, x1) if swap else (x0, y0, x1, y1), 1).contiguous()
    return turn


def _u(g, n, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(n, generator=g, device="cuda")


def _log_u(g, n, lo, hi):
    return torch.exp(_u(g, n, math.log(lo), math.log(hi)))


def _corners(g, n, clustered):
    """Lower-left corners: `clustered` of the n around 64 centres, the rest uniform, interleaved."""
    x, y = _u(g, n), _u(g, n)
    if clustered > 0:
        c = torch.rand(64, 2, generator=g, device="cuda")
        at = c[torch.randint(64, (n,), generator=g, device="cuda")]
        d = 0.02 * torch.randn(n, 2, generator=g, device="cuda")
        near = _u(g, n) < clustered
        x = torch.where(near, (at[:, 0] + d[:, 0]).clamp(0, 1), x)
        y = torch.where(near, (at[:, 1] + d[:, 1]).clamp(0, 1), y)
    return x, y


def _boxes(x, y, w, h):
    return torch.stack((x, y, x + w, y + h), 1).float().contiguous()


def _rects(g, n, data):
    x, y = _corners(g, n, 0.8 if data == "mixed" else 0.0)
    if data == "mixed":
        w, h = _log_u(g, n, SIDE_LO, SIDE_HI), _log_u(g, n, SIDE_LO, SIDE_HI)
    else:
        w, h = _u(g, n, 0, PLAIN_SIDE), _u(g, n, 0, PLAIN_SIDE)
    return _boxes(x, y, w, h)


def _renumber(g, r, rows):
    """Rows in another order: any, or (tiled) the 32 x 32 regions in any order and any order inside each."""
    r = r[_perm(g, r.shape[0])]
    if rows == "tiled":
        at = (r[:, :2] * 32).clamp(0, 31).long()
        r = r[torch.sort(_perm(g, 1024)[at[:, 1] * 32 + at[:, 0]], stable=True).indices]
    return r


def _queries(g, c):
    q, kind = c["q"], c["queries"]
    if kind == "selective":
        mean = (SIDE_HI - SIDE_LO) / math.log(SIDE_HI / SIDE_LO) if c["data"] == "mixed" else PLAIN_SIDE / 2
        w = h = (_log_u(g, q, c["sel_lo"], c["sel_hi"]).sqrt() - mean).clamp(min=0)
    elif kind == "small":
        w, h = _u(g, q, 0, 0.01), _u(g, q, 0, 0.01)
    elif kind == "windows":
        w, h = _u(g, q, 0.05, 0.2), _u(g, q, 0.05, 0.2)
    else:
        big = _u(g, q) < 0.01
        w = torch.where(big, _u(g, q, 0.05, 0.2), _u(g, q, 0, 1e-3))
        h = torch.where(big, _u(g, q, 0.05, 0.2), _u(g, q, 0, 1e-3))
    return _boxes(_u(g, q) * (1 - w), _u(g, q) * (1 - h), w, h)


def _hits_per_query(c):
    """Expected ids per query: the queries are uniform, so the data's clusters do not matter."""
    side = (SIDE_HI - SIDE_LO) / math.log(SIDE_HI / SIDE_LO) if c["data"] == "mixed" else PLAIN_SIDE / 2
    kind = c["queries"]
    if kind == "selective":
        p = (c["sel_hi"] - c["sel_lo"]) / math.log(c["sel_hi"] / c["sel_lo"]) + side * side / 4
    elif kind == "small":
        p = (0.005 + side) ** 2
    elif kind == "windows":
        p = (0.125 + side) ** 2
    else:
        p = 0.01 * (0.125 + side) ** 2 + 0.99 * (5e-4 + side) ** 2
    return c["n"] * min(1.0, p)


def _pairs(c):
    return c["n"] * c["m"] * JOIN_SIDE ** 2


def prepare(case, seed):
    c, base, g = case, _gen(_case_seed(case)), _gen(seed)
    s, turn = {"case": c}, _turn(g)
    if c["kind"] in ("join", "layers"):
        w = [_u(base, k, 0, JOIN_SIDE) for k in (c["n"], c["n"], c["m"], c["m"])]
        s["r"] = turn(_renumber(g, _boxes(*_corners(base, c["n"], 0.0), w[0], w[1]), "shuffled"))
        s["s"] = turn(_renumber(g, _boxes(*_corners(base, c["m"], 0.8), w[2], w[3]), "shuffled"))
        s["r_ids"] = torch.arange(c["n"], dtype=torch.int32, device="cuda")
        s["s_ids"] = torch.arange(c["m"], dtype=torch.int32, device="cuda")
        if c["kind"] == "join":
            s["trees"] = _two_trees(s)
        return s
    s["rects"] = turn(_renumber(g, _rects(base, c["n"], c["data"]), c["rows"]))
    s["ids"] = torch.arange(c["n"], dtype=torch.int32, device="cuda")
    s["queries"] = turn(_queries(base, c)[_perm(g, c["q"])])
    if c["kind"] == "build":
        return s
    s["tree"] = rt.RTree(s["rects"], s["ids"], fanout=c["fanout"], layout=c["layout"])
    del s["rects"], s["ids"]  # the tree has its own copy
    room = int(3 * c["q"] * _hits_per_query(c)) + 2 * c["n"]
    if c["kind"] == "plan":
        s["plan"] = rt.Plan(s["tree"], c["q"], room, mapping=c["mapping"])
    if c["kind"] == "host":
        s["queries"] = s["queries"].cpu().pin_memory()
        s["offsets"] = torch.empty(c["q"] + 1, dtype=torch.int64).pin_memory()
        s["out"] = torch.empty(room, dtype=torch.int32).pin_memory()
    return s


def _two_trees(s):
    c = s["case"]
    return (rt.RTree(s["r"], s["r_ids"], fanout=c["fanout"], layout=c["layout"], sort_children=c["sort_children"]),
            rt.RTree(s["s"], s["s_ids"], fanout=c["fanout_m"], layout=c["layout"],
                     sort_children=c["sort_children"]))


def _select(tree, s):
    c = s["case"]
    res = tree.range_select(s["queries"], unsorted=c["unsorted"], mapping=c["mapping"], order=c["order"])
    return {"offsets": res.offsets_tensor(), "ids": res.ids_tensor()}


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "select":
        return _select(s["tree"], s)
    if kind == "plan":
        s["plan"].run(s["queries"])
        return {"offsets": s["plan"].offsets_tensor(), "ids": s["plan"].ids_tensor()}
    if kind == "host":
        total = rt.rtree_range_select_host(s["tree"].handle, s["queries"], s["offsets"], s["out"],
                                           mapping=c["mapping"], order=c["order"])
        return {"offsets": s["offsets"], "ids": s["out"][:total]}
    if kind == "build":
        tree = rt.RTree(s["rects"], s["ids"], fanout=c["fanout"], layout=c["layout"])
        out = _select(tree, s)
        tree.close(torch.cuda.current_stream())
        return out
    r, t = s["trees"] if kind == "join" else _two_trees(s)
    out = {"pairs": r.join(t).ids_tensor()}
    if kind == "layers":
        r.close(torch.cuda.current_stream())
        t.close(torch.cuda.current_stream())
    return out


def work(case):
    """Bytes: every input that bears on the answer read once (a rectangle is 16 bytes and its id 4; no
    more of them than there are ids in the result), every output written once.  No arithmetic but
    comparisons."""
    c = case

    def tree_bytes(n, fanout):
        return n * 20 * (1 + 1 / (fanout - 1))

    if c["kind"] in ("join", "layers"):
        b = 20 * (c["n"] + c["m"]) + 8 * _pairs(c)
        if c["kind"] == "layers":  # rectangles in, trees out
            b += tree_bytes(c["n"], c["fanout"]) + tree_bytes(c["m"], c["fanout_m"])
        return {"bytes": b, "flops": 0}
    ids = c["q"] * _hits_per_query(c)
    b = 16 * c["q"] + 8 * (c["q"] + 1) + 4 * ids + 20 * min(c["n"], ids)
    if c["kind"] == "build":
        b += 20 * c["n"] + tree_bytes(c["n"], c["fanout"])
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    return None  # whole numbers only
