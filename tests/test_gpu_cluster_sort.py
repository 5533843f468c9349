"""Levels and sorts of the sizes at which the one-launch sort by a cluster starts, tiles its chunks and gives way to
the three-launch passes: the built tree equals the oracle's node by node, and ordered selects and joins stay exact."""
import numpy as np
import pytest

import oracle
from gpu_util import gpu_ready
from test_gpu_build import export_gpu
from test_oracle import random_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    return gpu_ready()


# 16 x 16384 = 2^18 items are one tile for each CTA of the cluster
@pytest.mark.parametrize("kind", ["uniform", "dups"])
@pytest.mark.parametrize("n,F", [(1024, 64), (1025, 64), (1025, 4), (1057, 128), (16 * 1024 + 1, 8), (2**18 - 31, 4),
                                 (2**18, 16), (2**18 + 1, 32), (2**19 - 1, 4), (2**19, 128), (2**19 + 1, 16),
                                 (2**19 + 1, 4), (2**21 + 1, 4), (4_200_000, 4)])  # slabs of 9, 10 and 11 bits
def test_tree(rt, n, F, kind):
    rects = random_case(kind, n, n)
    ids = np.arange(n, dtype=np.int32)[::-1].copy()
    got, _ = export_gpu(rt, rects, ids, F, "aos")
    want = oracle.Tree(rects, ids, F).export()
    for k in ("level_nodes", "counts", "leaf_ids", "mbrs"):
        assert np.array_equal(got[k], want[k]), k


def test_tree_of_equal_boxes(rt):  # every digit of every key the same; only the index decides
    rects = np.tile(np.array([[0.25, 0.5, 0.25, 0.5]], np.float32), (40_000, 1))
    got, _ = export_gpu(rt, rects, None, 16, "soa")
    want = oracle.Tree(rects, None, 16).export()
    for k in ("level_nodes", "counts", "leaf_ids", "mbrs"):
        assert np.array_equal(got[k], want[k]), k


@pytest.mark.parametrize("Q", [31, 1025, 2**18, 2**18 + 1])
def test_order_and_pairs(rt, Q):
    import torch
    rng = np.random.default_rng(Q)
    p = rng.random((500, 2), dtype=np.float32)
    q = rng.random((Q, 2), dtype=np.float32)
    rects, queries = np.concatenate([p, p + np.float32(0.05)], 1), np.concatenate([q, q], 1)
    with rt.RTree(rects, None, fanout=8) as t, rt.RTree(queries, None, fanout=8) as u:
        res = t.range_select(torch.from_numpy(queries).cuda(), order="hilbert")
        off, ids = res.to_numpy()
        res.close()
        res = u.join(t)
        pairs = res.to_numpy()[1]
        res.close()
    hit = (rects[:, 0] <= q[:, :1]) & (q[:, :1] <= rects[:, 2]) & (rects[:, 1] <= q[:, 1:]) & (q[:, 1:] <= rects[:, 3])
    i, j = np.nonzero(hit)
    assert np.array_equal(off, np.concatenate([[0], np.cumsum(hit.sum(1))])) and np.array_equal(ids, j)
    assert np.array_equal(pairs, np.stack([i, j], 1))
