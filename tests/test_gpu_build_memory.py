"""Builds where memory is short: 28 bytes a box of the largest level for its order, 4 for the order itself,
are what the sorts by passes over the whole chip take; the sorts of small levels have to do with that too."""
import numpy as np
import pytest

import oracle
from gpu_util import gpu_ready

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,fanout", [(1500, 128), (5000, 16), (150_000, 16), (500_000, 64), (524_288, 32)])
def test_build_in_little_memory(n, fanout):
    import torch
    rt = gpu_ready()
    rng = np.random.default_rng(n)
    p = rng.random((n, 2), dtype=np.float32)
    r = np.concatenate([p, p + np.float32(1e-3)], 1).astype(np.float32)
    q = np.concatenate([p[:50] - np.float32(0.02), p[:50] + np.float32(0.02)], 1).astype(np.float32)
    live, room = {}, 32 * n + 80_000

    def alloc(nbytes, stream):
        if sum(live.values()) + nbytes > room:
            return 0
        ptr = torch.cuda.caching_allocator_alloc(max(1, nbytes), None, stream)
        live[ptr] = nbytes
        return ptr

    def free(ptr, _stream):
        live.pop(ptr, None)
        torch.cuda.caching_allocator_delete(ptr)
    t = rt.RTree(torch.from_numpy(r).cuda(), None, fanout=fanout, allocator=rt.Allocator(alloc, free))
    ids = np.arange(n, dtype=np.int32)
    want = oracle.Tree(r, ids, fanout)
    got, ref = t.export(), want.export()
    assert np.array_equal(got["leaf_ids"], ref["leaf_ids"])
    room = 1 << 40
    res = t.range_select(q)
    off, found = res.to_numpy()
    res.close()
    w_off, w_ids = want.select(q)
    assert np.array_equal(off, w_off) and np.array_equal(found, w_ids)
    t.close()
    assert not live
