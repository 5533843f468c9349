"""A captured batch with more tasks of large queries than a plan has room for: those past the limit are walked
by one warp each, and the answers are the same."""
import numpy as np
import pytest

import oracle
from gpu_util import gpu_ready

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["soa", "aos", "lohi"])
def test_more_tasks_than_a_plan_holds(layout):
    import torch
    rt = gpu_ready()
    rng = np.random.default_rng(17)
    p = rng.random((400_000, 2), dtype=np.float32)
    r = np.concatenate([p, p], 1).astype(np.float32)
    lo = rng.random((2500, 2), dtype=np.float32) * np.float32(0.85)
    q = np.concatenate([lo, lo + np.float32(0.15)], 1).astype(np.float32)
    want = oracle.Tree(r, np.arange(len(r), dtype=np.int32), 4).select(q)
    with rt.RTree(torch.from_numpy(r).cuda(), None, fanout=4, layout=layout) as t:
        qc = torch.from_numpy(q).cuda()
        st = t.select_stats(qc)
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        # a task is reserved for every node above the leaves that a query visits; the plan holds 2^18, and the
        # batch is small enough for its large queries to be shared out
        assert st["nodes_visited"] - st["leaves_visited"] > 1 << 18
        assert 4 * st["leaves_visited"] < 4 * 160 * sms * 48
        plan = rt.Plan(t, len(q), len(want[1]) + 1000)
        for _ in range(2):
            plan.run(qc)
            off, ids = plan.to_numpy()
            assert np.array_equal(off, want[0]) and np.array_equal(ids, want[1])
        plan.close()
        res = t.range_select(qc)
        off, ids = res.to_numpy()
        res.close()
        assert np.array_equal(off, want[0]) and np.array_equal(ids, want[1])
