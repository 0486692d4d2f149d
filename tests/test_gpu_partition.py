"""GPU parity of the selection's partition by query at the edges of its tiles:
outputs of less than one tile to several, capacities that pick the smallest
and the largest super-tile, one query to the most a selection takes.  Lists
are whole numbers: equal to the oracle's, bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2203_14362_gb300 import datagen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402


# capacities: the output's own size (super-tiles of 1024 to 4096 pairs) and 20M (the largest super-tile)
@pytest.mark.parametrize("P,n,cap", [(1, 1023, 0), (1, 4097, 0), (3, 40_001, 0), (255, 30_000, 0), (256, 200_003, 0),
                                     (257, 200_003, 20_000_000), (1023, 100_001, 0), (1024, 150_000, 20_000_000)])
def test_partition_tiles(P, n, cap):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(P * 7 + n)
    box = 1 << 30
    rings = []
    for _ in range(P):  # overlapping rectangles of very uneven size; the first holds the whole box
        w, h = (rng.integers(1, box // 3, 2) * rng.random(2) ** 3).astype(np.int64) + 1
        x, y = rng.integers(0, box - w), rng.integers(0, box - h)
        rings.append(g.rect_polygon(x, y, x + w, y + h))
    rings[0] = g.rect_polygon(0, 0, box, box)
    v = np.concatenate(rings)
    o = np.arange(0, 4 * (P + 1), 4, dtype=np.uint64)
    pts = g.uniform_points(n, P)
    pr = oracle.Prepared(v, o)
    want_ids, want_off = pr.select(pts)
    pr.close()
    eng = spx.Engine(0)
    try:
        dpts = torch.from_numpy(pts).cuda()
        ph = eng.load_points(dpts)
        ih = eng.build_index(eng.load_polygons(v, o), grid_log2=7)
        ids = torch.full((cap or want_ids.shape[0],), -1, dtype=torch.int32, device="cuda")
        offs = torch.zeros(P + 1, dtype=torch.int64, device="cuda")
        for _ in range(2):  # run directly, then replayed
            ids.fill_(-1)
            m = eng.select(ph, ih, ids, offs)
            assert m == want_ids.shape[0]
            assert np.array_equal(offs.cpu().numpy().view(np.uint64), want_off)
            assert np.array_equal(ids[:m].cpu().numpy().view(np.uint32), want_ids)
            assert bool((ids[m:] == -1).all())
    finally:
        eng.close()
