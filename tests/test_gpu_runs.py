"""Neighbouring whole subtrees are taken as one run: windows over trees of every fanout and layout, sorted and
unsorted, and over a loaded tree whose siblings' entries do not follow one another, against brute force."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_csr_equal, gpu_ready
from persist_util import HEADER_BYTES, reseal
from test_oracle import random_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    return gpu_ready()


def windows(seed):
    rng = np.random.default_rng(seed)
    lo = rng.random((300, 2)).astype(np.float32)
    side = np.float32(0.5) * rng.random((300, 2)).astype(np.float32) ** 2
    return np.concatenate([np.concatenate([lo, lo + side], 1), np.array([[-1, -1, 2, 2]], np.float32)])


def select_np(t, q, unsorted=False):
    res = t.range_select(q, unsorted)
    off, ids = res.to_numpy()
    res.close()
    return off, np.concatenate([np.sort(s) if unsorted else s for s in np.split(ids, off[1:-1])])


@pytest.mark.parametrize("layout", ["soa", "aos", "lohi"])
@pytest.mark.parametrize("F", [4, 8, 16, 32, 64, 128])
def test_runs(rt, F, layout):
    rects, q = random_case("uniform", 9001, F), windows(F)
    want = oracle.brute_select(rects, q, None)
    with rt.RTree(rects, None, fanout=F, layout=layout) as t:
        assert_csr_equal(select_np(t, q), want)
        assert_csr_equal(select_np(t, q, True), want)


@pytest.mark.parametrize("F", [4, 16, 32, 64])
def test_siblings_out_of_entry_order(rt, F, tmp_path):
    n = F * F * 3  # at least three internal nodes, full leaves
    rects, q = random_case("uniform", n, 7), windows(7)
    with rt.RTree(rects, None, fanout=F, layout="aos", sort_children=False) as t:
        t.save(str(tmp_path / "t.rtree"))
        M, level = t.info()["nodes"], t.export()["level_nodes"]
    buf = bytearray((tmp_path / "t.rtree").read_bytes())
    ends = HEADER_BYTES + np.cumsum([0, M * F * 16, M * 16, M * 16])
    mbr, meta, nbox = [np.frombuffer(buf, ty, (b - a) // 4, a).reshape(M, -1, 4)
                       for ty, a, b in zip((np.float32, np.int32, np.float32), ends[:-1], ends[1:])]
    parent = sum(level[:-3]) if len(level) > 2 else 0  # first node two levels above the leaves
    g = int(meta[parent, 0, 0])
    assert meta[parent, 0, 1] >= 2
    for a in (mbr, meta, nbox):  # its first two children change places
        a[[g, g + 1]] = a[[g + 1, g]]
    mbr[parent, [0, 1]] = mbr[parent, [1, 0]]
    assert meta[g, 0, 3] != meta[g + 1, 0, 2]
    (tmp_path / "u.rtree").write_bytes(bytes(reseal(buf)))
    want = oracle.brute_select(rects, q, None)
    with rt.RTree.load(str(tmp_path / "u.rtree")) as t:
        assert_csr_equal(select_np(t, q), want)
        assert_csr_equal(select_np(t, q, True), want)
