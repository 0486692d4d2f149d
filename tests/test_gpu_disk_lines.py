"""GPU parity of distance queries on both sides of the lines of their pass 1: 2048 and
2049 disks (two kernels or one for joins), 11776 and 11777 (counters in shared or in
global memory), a table within and above the small-join limit, points crowded into
many disks, outputs above and below the emit pass's stage, the smallest grids (whose
cover bitmap is less than a word), counts on both sides of 2^23 points.  Whole numbers: equal to the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2203_14362_gb300 import datagen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402

BOX = 1 << 30
LIMIT = 4096 * 256


def case(q, n):
    rng = np.random.default_rng(q)
    c = rng.integers(0, BOX, (q, 2))
    r = rng.integers(0, 1 << 23, q)
    c[: q // 20] = BOX // 2 + rng.integers(-(1 << 20), 1 << 20, (q // 20, 2))  # many around one place
    pts = g.uniform_points(n, q)
    pts[::9] = BOX // 2 + (pts[::9] >> 9)
    pts[::777] = -3
    return c.astype(np.int32), r.astype(np.int32), pts


@pytest.mark.parametrize("q,n,gl", [(2048, 20_011, 0), (2049, 20_011, 0), (2049, LIMIT + 1, 0), (2048, LIMIT + 1, 7),
                                    (11776, 10_007, 0), (11777, 10_007, 0), (700, 30_001, 1), (2500, 30_001, 2)])
def test_disk_lines(q, n, gl):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c, r, pts = case(q, n)
    want, want_counts = oracle.disk_join(pts, c, r)
    eng = spx.Engine(0)
    try:
        dpts = torch.from_numpy(pts).cuda()
        ph = eng.load_points(dpts)
        ih = eng.build_disk_index(c, r, gl)
        for cap in (want.shape[0], want.shape[0] // 2):
            pairs = torch.full((want.shape[0], 2), -1, dtype=torch.int32, device="cuda")
            counts = torch.full((q,), 7, dtype=torch.int64, device="cuda")
            total = torch.zeros(1, dtype=torch.int64, device="cuda")
            eng.join(ph, ih, pairs[:cap], counts, total=total, sync=False)
            torch.cuda.synchronize()
            got = pairs.cpu().numpy().view(np.uint32)
            assert total.item() == want.shape[0]
            assert np.array_equal(got[:cap], want[:cap]) and (got[cap:] == 0xFFFFFFFF).all()
            assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
        eng.join(ph, ih, pairs, None, total=total, sync=False)  # without counts
        torch.cuda.synchronize()
        assert np.array_equal(pairs.cpu().numpy().view(np.uint32), want)
        for table in (ph, eng.cluster_points(ph)):
            counts.fill_(7)
            eng.aggregate(table, ih, counts)
            assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
        if q <= 1024:
            ids = torch.empty(want.shape[0], dtype=torch.int32, device="cuda")
            offs = torch.empty(q + 1, dtype=torch.int64, device="cuda")
            assert eng.select(ph, ih, ids, offs) == want.shape[0]
            order = np.argsort(want[:, 1], kind="stable")
            assert np.array_equal(ids.cpu().numpy().view(np.uint32), want[order, 0])
    finally:
        eng.close()


@pytest.mark.parametrize("n", [1 << 23, (1 << 23) + 1])
def test_disk_count_lines(n):  # one pass, or the join's two
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c, r, pts = case(60, n)
    want = oracle.disk_join(pts, c, r)[1]
    eng = spx.Engine(0)
    try:
        dpts = torch.from_numpy(pts).cuda()
        ph = eng.load_points(dpts)
        ih = eng.build_disk_index(c, r)
        counts = torch.full((60,), 7, dtype=torch.int64, device="cuda")
        eng.aggregate(ph, ih, counts)
        assert np.array_equal(counts.cpu().numpy().view(np.uint64), want)
    finally:
        eng.close()
