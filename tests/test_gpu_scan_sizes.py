"""Batches of the sizes at which the counts' scans fit one tile, one launch and several: offsets and ids against brute
force, for the sorted, unsorted, work-queue, captured and host-result forms."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_csr_equal, gpu_ready
from test_oracle import random_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    return gpu_ready()


@pytest.mark.parametrize("Q", [1, 7, 8, 9, 2047, 2048, 2049, 4097])
def test_offsets(rt, Q):
    rects, q = random_case("uniform", 3000, 11), random_case("uniform", Q, Q)
    want = oracle.brute_select(rects, q, None)
    with rt.RTree(rects, None, fanout=16) as t:
        for kw in ({}, {"order": "hilbert"}, {"mapping": "work_queue"}, {"unsorted": True}):
            res = t.range_select(q, **kw)
            off, ids = res.to_numpy()
            res.close()
            if kw.get("unsorted"):
                ids = np.concatenate([np.sort(s) for s in np.split(ids, off[1:-1])])
            assert_csr_equal((off, ids), want)
        plan = rt.Plan(t, Q, len(want[1]) + 1)
        plan.run(q)
        assert_csr_equal(plan.to_numpy(), want)
        plan.close()
        off, ids = np.zeros(Q + 1, np.int64), np.zeros(max(1, len(want[1])), np.int32)
        total = rt.rtree_range_select_host(t.handle, q, off, ids)
        assert_csr_equal((off, ids[:total]), want)
