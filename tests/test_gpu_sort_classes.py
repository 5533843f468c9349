"""The segmented sort at the edges of its size classes, for ids of several kinds.

A tree of exactly n rectangles is asked for all of them (one run of ids), for
those left of a cut (runs and leaf hits) and for one; the ids returned have to
be the sorted ids of a NumPy comparison, bit for bit.
"""
import numpy as np
import pytest

from gpu_util import gpu_ready, select_gpu

pytestmark = pytest.mark.gpu

# 252 ids per warp and eight ids a lane: the CTA sorts end at these sizes
EDGES = [256, 1008, 2016, 4032, 8064, 16128, 32256]


@pytest.fixture(scope="module")
def rt():
    return gpu_ready()


def make_ids(kind, n, rng):
    if kind == "shuffled":
        return rng.permutation(n).astype(np.int32) - np.int32(n // 3)
    if kind == "sparse":  # the whole range of int32
        return rng.integers(-2**31, 2**31 - 1, n, dtype=np.int64, endpoint=True).astype(np.int32)
    if kind == "bands":  # a few dense bands far apart
        return (rng.integers(0, 7, n) * 50_000_000 + rng.permutation(n) // 2).astype(np.int32)
    if kind == "repeated":  # every id several times, some very often
        return np.where(rng.random(n) < 0.1, 5, rng.permutation(n) // 4).astype(np.int32)
    return np.full(n, np.iinfo(np.int32).max, np.int32)  # "equal"


@pytest.mark.parametrize("kind", ["shuffled", "sparse", "bands", "repeated", "equal"])
@pytest.mark.parametrize("n", sorted({e + d for e in EDGES for d in (0, 1)} | {2, 33, 257, 40_003, 150_001}))
def test_sorted_at_class_edges(rt, n, kind):
    rng = np.random.default_rng(n)
    x, y = rng.random(n, dtype=np.float32), rng.random(n, dtype=np.float32)
    rects = np.stack([x, y, x + np.float32(1e-4), y + np.float32(1e-4)], 1).astype(np.float32)
    ids = make_ids(kind, n, rng)
    queries = np.array([[-1, -1, 3, 3], [-1, -1, 0.7, 3], [rects[0, 0], rects[0, 1], rects[0, 2], rects[0, 3]]],
                       np.float32)
    want = [np.sort(ids[(rects[:, 0] <= q[2]) & (q[0] <= rects[:, 2]) & (rects[:, 1] <= q[3]) & (q[1] <= rects[:, 3])])
            for q in queries]
    for fanout, layout, mapping in ((64, "aos", "auto"), (16, "soa", "auto"), (32, "lohi", "work_queue")):
        off, got = select_gpu(rt, rects, ids, queries, fanout=fanout, layout=layout, mapping=mapping)
        for i, w in enumerate(want):
            assert np.array_equal(got[off[i]:off[i + 1]], w), (n, kind, fanout, i)
