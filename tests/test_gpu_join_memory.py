"""The join by levels where memory is short, and where a level has more node pairs than its buffer."""
import numpy as np
import pytest

import oracle
from gpu_util import gpu_ready

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    return gpu_ready()


def boxes(rng, n, side):
    p = rng.random((n, 2), dtype=np.float32)
    return np.concatenate([p, p + np.float32(side) * rng.random((n, 2), dtype=np.float32)], 1).astype(np.float32)


def limited(rt):
    """An allocator that hands out at most limit["bytes"] at a time."""
    import torch
    live, limit = {}, {"bytes": 1 << 40}

    def alloc(nbytes, stream):
        if sum(live.values()) + nbytes > limit["bytes"]:
            return 0
        p = torch.cuda.caching_allocator_alloc(max(1, nbytes), None, stream)
        live[p] = nbytes
        return p

    def free(p, _stream):
        live.pop(p, None)
        torch.cuda.caching_allocator_delete(p)
    return rt.Allocator(alloc, free), live, limit


# A join by counting first takes 32 bytes a result in the sort of its pairs, 20 bytes a node pair of the
# last level beside them, and the digit counts of a large sort (1.3 MB); that much has to do.
@pytest.mark.parametrize("n,side,fanout", [(1000, 0.001, 16), (5000, 0.2, 16), (5000, 0.1, 4), (200_000, 0.005, 32)])
@pytest.mark.parametrize("sort_children", [False, True])
def test_join_in_little_memory(rt, n, side, fanout, sort_children):
    rng = np.random.default_rng(n)
    r, s = boxes(rng, n, side), boxes(rng, n, side)
    A, live, limit = limited(rt)
    a = rt.RTree(r, None, fanout=fanout, layout="aos", sort_children=sort_children, allocator=A)
    b = rt.RTree(s, None, fanout=fanout, layout="aos", sort_children=sort_children, allocator=A)
    res = a.join(b)
    want = res.to_numpy()[1]
    res.close()
    if n <= 5000:
        ids = np.arange(n, dtype=np.int32)
        assert np.array_equal(want, oracle.Tree(r, ids, fanout).join(oracle.Tree(s, ids, fanout)))
    trees = sum(live.values())
    node_pairs = rt.rtree_join_stats(a.handle, b.handle)["pairs_leaf"]
    limit["bytes"] = trees + 32 * len(want) + 20 * node_pairs + (1_300_000 if len(want) > 1 << 18 else 2000)
    for _ in range(2):
        res = a.join(b)
        assert np.array_equal(res.to_numpy()[1], want)
        res.close()
    limit["bytes"] = trees + 1000
    with pytest.raises(rt.RTreeError) as e:
        a.join(b)
    assert e.value.status == rt.RTREE_ENOMEM
    assert sum(live.values()) == trees
    a.close()
    b.close()
    assert not live


# 3000 boxes at F = 4 have 750 leaves, most of which meet: more than the 8 node pairs a node and 65536 of a level's buffer
@pytest.mark.parametrize("sort_children", [False, True])
def test_level_outgrown(rt, sort_children):
    rng = np.random.default_rng(11)
    r, s = boxes(rng, 3000, 0.8), boxes(rng, 3000, 0.8)
    ids = np.arange(3000, dtype=np.int32)
    want = oracle.Tree(r, ids, 4).join(oracle.Tree(s, ids, 4))
    with rt.RTree(r, ids, fanout=4, sort_children=sort_children) as a, \
            rt.RTree(s, ids, fanout=4, sort_children=sort_children) as b:
        st = rt.rtree_join_stats(a.handle, b.handle)
        assert st["pairs_leaf"] > 8 * (a.info()["nodes"] + b.info()["nodes"]) + 65536 and st["pairs_found"] == len(want)
        res = a.join(b)
        _, got = res.to_numpy()
        res.close()
    assert np.array_equal(got, want)
