"""Queries large enough to be shared out among warps, beside small ones: every fanout and layout, trees of one
level and more, called and captured, against a NumPy comparison."""
import numpy as np
import pytest

from gpu_util import gpu_ready

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    return gpu_ready()


@pytest.mark.parametrize("layout", ["soa", "aos", "lohi"])
@pytest.mark.parametrize("F", [4, 8, 16, 32, 64, 128])
@pytest.mark.parametrize("n", [100, 4095, 30_011])
def test_windows(rt, F, layout, n):
    import torch
    rng = np.random.default_rng(n + F)
    p = rng.random((n, 2), dtype=np.float32)
    rects = np.concatenate([p, p + np.float32(0.002) * rng.random((n, 2), dtype=np.float32)], 1).astype(np.float32)
    ids = rng.permutation(n).astype(np.int32)
    # thin bands cut many leaves and hold few whole ones; windows hold many; the last ones are small
    q = np.array([[0.1, 0.1, 0.9, 0.9], [0.0, 0.4, 1.0, 0.45], [0.3, 0, 0.31, 1], [-1, -1, 2, 2], [0.5, 0.5, 0.5, 0.5]],
                 np.float32)
    q = np.concatenate([q, np.tile(np.array([[0.2, 0.2, 0.201, 0.201]], np.float32), (40, 1))])
    want = [np.sort(ids[(rects[:, 0] <= w[2]) & (w[0] <= rects[:, 2]) & (rects[:, 1] <= w[3]) & (w[1] <= rects[:, 3])])
            for w in q]
    total = sum(len(w) for w in want)
    with rt.RTree(torch.from_numpy(rects).cuda(), torch.from_numpy(ids).cuda(), fanout=F, layout=layout) as t:
        for order in ("input", "hilbert"):
            res = t.range_select(torch.from_numpy(q).cuda(), order=order)
            off, got = res.to_numpy()
            res.close()
            for i, w in enumerate(want):
                assert np.array_equal(got[off[i]:off[i + 1]], w), (order, i)
        plan = rt.Plan(t, 64, 4 * total + 64 * F)
        for _ in range(2):
            assert plan.run(q) == total
            off, got = plan.to_numpy()
            for i, w in enumerate(want):
                assert np.array_equal(got[off[i]:off[i + 1]], w), i
        plan.close()
        small = rt.Plan(t, 64, max(1, total // 2))  # the size needed is reported past the large queries too
        with pytest.raises(rt.RTreeError) as e:
            small.run(q)
        assert e.value.status == rt.RTREE_EOVERFLOW
        small.close()
