"""GPU parity of distance queries where their kernels change path: the join and
selection on both sides of the small-table limit (1,048,576 points), the count
on both sides of its two-pass limit (2,097,152) in row order and over the
clustered copy, an index whose block summary resolves little, and 32-bit
per-point results (more than 65534 disks) with points in more disks than a
result stores.  Whole numbers: equal to the oracle's, bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2203_14362_gb300 import datagen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402

LIMIT = 4096 * 256


def disks(name):
    rng = np.random.default_rng(5)
    if name == "many":  # 65000 small ones, and 1100 around one place
        c = np.concatenate([rng.integers(0, 1 << 30, (65000, 2)), np.full((1100, 2), 1 << 21)])
        r = np.concatenate([rng.integers(0, 1 << 20, 65000), rng.integers(1 << 20, 1 << 21, 1100)])
    elif name == "dense":  # most blocks of the box hold a boundary
        c, r = rng.integers(0, 1 << 30, (60, 2)), rng.integers(1 << 26, 1 << 28, 60)
    else:
        c, r = rng.integers(0, 1 << 30, (40, 2)), rng.integers(0, 1 << 25, 40)
    return c.astype(np.int32), r.astype(np.int32)


@pytest.mark.parametrize("name,n", [("few", LIMIT), ("few", LIMIT + 1), ("dense", LIMIT + 1), ("many", 20_001)])
def test_disk_join_paths(name, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c, r = disks(name)
    pts = g.uniform_points(n, 3)
    if name == "many":
        pts[::40] >>= 8
    want, want_counts = oracle.disk_join(pts, c, r)
    eng = spx.Engine(0)
    try:
        dpts = torch.from_numpy(pts).cuda()
        ph = eng.load_points(dpts)
        for on_device in (False, True):
            ih = eng.build_disk_index(c, r, 0 if name != "dense" else 6, on_device=on_device)
            pairs = torch.empty((want.shape[0], 2), dtype=torch.int32, device="cuda")
            counts = torch.full((len(r),), 7, dtype=torch.int64, device="cuda")
            m = eng.join(ph, ih, pairs, counts)
            assert m == want.shape[0]
            assert np.array_equal(pairs.cpu().numpy().view(np.uint32), want)
            assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
            if len(r) <= 1024:
                ids = torch.empty(m, dtype=torch.int32, device="cuda")
                offs = torch.empty(len(r) + 1, dtype=torch.int64, device="cuda")
                assert eng.select(ph, ih, ids, offs) == m
                order = np.argsort(want[:, 1], kind="stable")
                assert np.array_equal(ids.cpu().numpy().view(np.uint32), want[order, 0])
                assert np.array_equal(offs.cpu().numpy()[1:], np.cumsum(want_counts.astype(np.int64)))
            eng.free(ih)
    finally:
        eng.close()


@pytest.mark.parametrize("n", [2 * LIMIT, 2 * LIMIT + 257])
def test_disk_count_paths(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c, r = disks("few")
    pts = g.mixture_points(n, 3)
    pts[::999] = -7
    want = oracle.disk_join(pts, c, r)[1]
    eng = spx.Engine(0)
    try:
        dpts = torch.from_numpy(pts).cuda()
        ph = eng.load_points(dpts)
        ih = eng.build_disk_index(c, r)
        counts = torch.empty(len(r), dtype=torch.int64, device="cuda")
        for table in (ph, eng.cluster_points(ph)):
            counts.fill_(7)
            eng.aggregate(table, ih, counts)
            assert np.array_equal(counts.cpu().numpy().view(np.uint64), want)
    finally:
        eng.close()
