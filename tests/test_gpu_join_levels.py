"""The join by levels where its buffers and node tests can go wrong: results past the first buffer, many
children on both sides, trees of unequal height, against an all-pairs NumPy comparison."""
import numpy as np
import pytest

from gpu_util import gpu_ready

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    return gpu_ready()


def boxes(rng, n, side):
    p = rng.random((n, 2), dtype=np.float32)
    return np.concatenate([p, p + np.float32(side) * rng.random((n, 2), dtype=np.float32)], 1).astype(np.float32)


def all_pairs(r, s, rid, sid):
    hit = ((r[:, None, 0] <= s[None, :, 2]) & (s[None, :, 0] <= r[:, None, 2]) &
           (r[:, None, 1] <= s[None, :, 3]) & (s[None, :, 1] <= r[:, None, 3]))
    i, j = np.nonzero(hit)
    p = np.stack([rid[i], sid[j]], 1)
    return p[np.lexsort((p[:, 1], p[:, 0]))]


# sides of 1 make every pair qualify somewhere near: 2000 x 1500 boxes give more pairs than the first buffer holds
@pytest.mark.parametrize("n,m,side", [(1, 1, 1.0), (2000, 1500, 1.0), (129, 3000, 0.1), (3000, 5, 0.02), (4097, 4095, 0.01)])
@pytest.mark.parametrize("fr,fs", [(4, 128), (16, 16), (128, 128), (32, 8)])
@pytest.mark.parametrize("sort_children", [False, True])
def test_join_pairs(rt, n, m, side, fr, fs, sort_children):
    rng = np.random.default_rng(n + m)
    r, s = boxes(rng, n, side), boxes(rng, m, side)
    rid = rng.integers(-2**31, 2**31 - 1, n).astype(np.int32)
    sid = np.arange(m, dtype=np.int32) - 7
    want = all_pairs(r, s, rid, sid)
    with rt.RTree(r, rid, fanout=fr, layout="soa", sort_children=sort_children) as a, \
            rt.RTree(s, sid, fanout=fs, layout="aos", sort_children=sort_children) as b:
        res = a.join(b)
        _, got = res.to_numpy()
        res.close()
        assert rt.rtree_join_stats(a.handle, b.handle)["pairs_found"] == len(want)
    assert np.array_equal(got, want)
