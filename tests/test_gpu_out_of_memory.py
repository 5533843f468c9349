"""Calls that run out of device memory: RTREE_ENOMEM, and nothing else is disturbed."""
import threading

import numpy as np
import pytest

from gpu_util import gpu_ready

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["thread_local", "relaxed"])
def test_another_threads_capture_goes_on(mode):
    import torch
    rt = gpu_ready()
    rng = np.random.default_rng(1)
    p = rng.random((1_000_000, 2), dtype=np.float32)
    t = rt.RTree(torch.from_numpy(np.concatenate([p, p], 1)).cuda())
    everything = torch.tensor([[-1.0, -1.0, 2.0, 2.0]], device="cuda").repeat(300_000, 1).contiguous()  # 1.2 TB of ids
    side, stream = torch.cuda.Stream(), torch.cuda.Stream()
    t.range_select(everything[:10], stream=side).close()
    x = torch.zeros(1000, device="cuda")
    torch.cuda.synchronize()
    out = []

    def body():
        try:
            t.range_select(everything, stream=side).close()
            out.append(None)
        except rt.RTreeError as e:
            out.append(e)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        g.capture_begin(capture_error_mode=mode)
        x.add_(1)
        th = threading.Thread(target=body)
        th.start()
        th.join()
        x.add_(1)
        g.capture_end()
        g.replay()
    torch.cuda.synchronize()
    assert out[0] is not None and out[0].status == rt.RTREE_ENOMEM, out[0]
    assert float(x.sum()) == 2000
    res = t.range_select(everything[:10])
    assert res.total == 10_000_000
    res.close()
    t.close()
