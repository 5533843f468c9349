"""What a plan takes from its tree's allocator: a fixed part of the queries and ids it can hold, and no more than
the work queue's items besides, with either mapping."""
import numpy as np
import pytest

import oracle
from gpu_util import gpu_ready
from paper_2309_16913_gb300 import datagen as dg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mapping", ["warp_per_query", "work_queue"])
@pytest.mark.parametrize("q,fanout", [(1, 16), (500, 64), (3000, 4)])
def test_plan_memory(mapping, q, fanout):
    import torch
    rt = gpu_ready()
    w = dg.workload("plain", n=50_000, q=q)
    want = oracle.Tree(w.rects, w.ids, fanout).select(w.queries)
    inner, taken = rt.TorchAllocator(), []

    def alloc(nbytes, stream):
        taken.append(nbytes)
        return inner._alloc(nbytes, stream)
    t = rt.RTree(torch.from_numpy(w.rects).cuda(), torch.from_numpy(w.ids).cuda(), fanout=fanout,
                 allocator=rt.Allocator(alloc, inner._free))
    ids = max(1, len(want[1])) + 1000
    taken.clear()
    plan = rt.Plan(t, q, ids, mapping=mapping)
    slots = 2 * ids + 4 * fanout * q
    assert sum(taken) <= 60 * q + 4 * slots + 12 * ids + 8 * (q + (1 << 20)) + 18 * 256
    queries = torch.from_numpy(w.queries).cuda()
    for k in (q, 1, max(1, q // 2)):
        plan.run(queries[:k])
        off, got = plan.to_numpy()
        assert np.array_equal(off, want[0][:k + 1]) and np.array_equal(got, want[1][:want[0][k]])
    plan.close()
    t.close()
