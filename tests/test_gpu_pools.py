"""Where large results live without an allocator: in the library's pool, which rtree_trim empties, or in the
caller's as soon as the caller manages the default pool or sets one of its own."""
import ctypes as C

import numpy as np
import pytest

from gpu_util import gpu_ready

pytestmark = pytest.mark.gpu

THRESHOLD, POOL_OF_POINTER = 4, 17  # CU_MEMPOOL_ATTR_RELEASE_THRESHOLD, CU_POINTER_ATTRIBUTE_MEMPOOL_HANDLE
MB = 1 << 20


class PoolProps(C.Structure):
    _fields_ = [("alloc_type", C.c_int), ("handle_types", C.c_int), ("loc_type", C.c_int), ("loc_id", C.c_int),
                ("security", C.c_void_p), ("max_size", C.c_size_t), ("rest", C.c_ubyte * 56)]


@pytest.fixture(scope="module")
def env():
    import torch
    rt = gpu_ready()
    cu = C.CDLL("libcuda.so.1")
    torch.zeros(1, device="cuda")
    p = np.random.default_rng(1).random((1_000_000, 2), dtype=np.float32)
    t = rt.RTree(torch.from_numpy(np.concatenate([p, p], 1)).cuda())
    q = torch.tensor([[-1.0, -1.0, 2.0, 2.0]], device="cuda").repeat(400, 1).contiguous()  # 1.6 GB of ids
    t.range_select(q).close()
    default = C.c_void_p()
    assert cu.cuDeviceGetDefaultMemPool(C.byref(default), 0) == 0
    yield rt, torch, cu, t, q, default
    t.close()


def pool_of(cu, ptr):
    h = C.c_void_p()
    assert cu.cuPointerGetAttribute(C.byref(h), POOL_OF_POINTER, C.c_uint64(ptr)) == 0
    return h.value


def idle_memory(env):
    """Free memory once the default pool keeps nothing."""
    rt, torch, cu, t, q, default = env
    torch.cuda.synchronize()
    assert cu.cuMemPoolTrimTo(default, C.c_size_t(0)) == 0
    return torch.cuda.mem_get_info()[0]


def select(env):
    """One large select: the pool of its ids."""
    rt, torch, cu, t, q, default = env
    res = t.range_select(q).wait()
    h = pool_of(cu, rt.rtree_result_ids(res.handle))
    res.close()
    return h


def test_trim_gives_results_back(env):
    rt, default = env[0], env[5]
    rt.rtree_trim()
    before = idle_memory(env)
    assert select(env) != default.value
    kept = idle_memory(env)
    rt.rtree_trim()
    after = idle_memory(env)
    assert before - kept > 1500 * MB and before - after < 100 * MB
    with pytest.raises(rt.RTreeError):
        rt.rtree_trim(99)


def test_callers_release_threshold(env):
    rt, torch, cu, t, q, default = env
    old = C.c_uint64()
    assert cu.cuMemPoolGetAttribute(default, THRESHOLD, C.byref(old)) == 0
    rt.rtree_trim()
    before = idle_memory(env)
    select(env)  # kept in the library's pool
    assert cu.cuMemPoolSetAttribute(default, THRESHOLD, C.byref(C.c_uint64(0))) == 0
    try:
        assert select(env) == default.value
        assert before - idle_memory(env) < 100 * MB  # the library's pool keeps nothing either
    finally:
        assert cu.cuMemPoolSetAttribute(default, THRESHOLD, C.byref(old)) == 0
    assert select(env) != default.value


def test_callers_pool(env):
    rt, torch, cu, t, q, default = env
    mine, props = C.c_void_p(), PoolProps(alloc_type=1, loc_type=1, loc_id=0)
    assert cu.cuMemPoolCreate(C.byref(mine), C.byref(props)) == 0
    assert cu.cuDeviceSetMemPool(0, mine) == 0
    try:
        assert select(env) == mine.value
    finally:
        assert cu.cuDeviceSetMemPool(0, default) == 0
        torch.cuda.synchronize()
        assert cu.cuMemPoolDestroy(mine) == 0
    assert select(env) not in (mine.value, default.value)
