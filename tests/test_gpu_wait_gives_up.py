"""Work-queue passes that give up with work left undone.

With a wait limit of one cycle the warps that find no work leave at once, and what busy warps then hand
over is never taken: a descriptor pass leaves slots unset, and after a count pass the next one finds too
few of them.  The call reports RTREE_ETIMEOUT, the sort leaves the incomplete queries out, and later calls
are exact.  Windows of all sizes, so that each way of gathering ids meets incomplete queries.
"""
import threading
import time

import numpy as np
import pytest

import oracle
from gpu_util import gpu_ready
from paper_2309_16913_gb300 import datagen as dg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def data():
    import torch
    rt = gpu_ready()
    w = dg.workload("plain", n=300_000, q=10)
    rng = np.random.default_rng(3)
    side = rng.choice([0.01, 0.03, 0.1, 0.3, 0.7], 120).astype(np.float32)
    lo = (rng.random((120, 2)) * (1 - side[:, None])).astype(np.float32)
    queries = np.concatenate([lo, lo + side[:, None]], 1).astype(np.float32)
    want = oracle.Tree(w.rects, w.ids, 16).select(queries)
    lens = np.diff(want[0])
    assert (lens <= 256).any() and ((lens > 256) & (lens <= 32256)).any() and (lens > 32256).any()
    t = rt.RTree(torch.from_numpy(w.rects).cuda(), torch.from_numpy(w.ids).cuda(), fanout=16)
    q = torch.from_numpy(queries).cuda()
    exact(t, q, want)  # the kernels are loaded, so that a call's launches do not wait for the stream
    yield rt, t, q, want
    t.close()


def exact(t, q, want):
    for mapping in ("work_queue", "warp_per_query"):
        res = t.range_select(q, mapping=mapping)
        off, ids = res.to_numpy()
        res.close()
        assert np.array_equal(off, want[0]) and np.array_equal(ids, want[1]), mapping


def second_pass_gives_up(rt, call):
    """Runs `call` with the limit lowered for its second pass: the stream is held while the first one is
    enqueued, so that the call waits for it."""
    import torch
    out = []

    def body():
        try:
            out.append(call())
        except rt.RTreeError as e:
            out.append(e)
    torch.cuda.synchronize()
    torch.cuda._sleep(1_000_000_000)  # about half a second
    before = rt.rtree_launch_count()
    th = threading.Thread(target=body)
    th.start()
    until = time.monotonic() + 0.3
    while rt.rtree_launch_count() < before + 2 and time.monotonic() < until:  # the queue and the count pass
        time.sleep(0.001)
    rt.rtree_debug_wq_wait(1, hold=False)
    th.join()
    assert isinstance(out[0], rt.RTreeError) and out[0].status == rt.RTREE_ETIMEOUT, out[0]
    assert "count pass" not in str(out[0])


def test_descriptor_pass(data):
    rt, t, q, want = data
    for _ in range(3):
        def call():
            res = t.range_select(q, mapping="work_queue")
            try:
                return res.to_numpy()
            finally:
                res.close()
        second_pass_gives_up(rt, call)
        exact(t, q, want)


def test_descriptor_pass_to_host(data):
    import torch
    rt, t, q, want = data
    off = torch.zeros(q.shape[0] + 1, dtype=torch.int64).pin_memory()
    ids = torch.zeros(len(want[1]), dtype=torch.int32).pin_memory()
    def call():
        rt.rtree_range_select_host(t.handle, q, off, ids, mapping="work_queue")
    call()
    second_pass_gives_up(rt, call)
    assert np.array_equal(off.numpy(), want[0])
    exact(t, q, want)


def test_count_pass_of_a_plan(data):
    rt, t, q, want = data
    plan = rt.Plan(t, q.shape[0], len(want[1]) + 1000, mapping="work_queue")
    rt.rtree_debug_wq_wait(1, hold=False)  # the plan's first run captures its graph with this limit
    for _ in range(3):
        with pytest.raises(rt.RTreeError) as e:
            plan.run(q)
        assert e.value.status == rt.RTREE_ETIMEOUT, str(e.value)
    plan.close()
    plan = rt.Plan(t, q.shape[0], len(want[1]) + 1000, mapping="work_queue")
    plan.run(q)
    off, ids = plan.to_numpy()
    plan.close()
    assert np.array_equal(off, want[0]) and np.array_equal(ids, want[1])
    exact(t, q, want)
