"""GPU parity of buffered-polygon queries where their kernels change path: the
join and selection on both sides of the small-table limit (1,048,576 points),
the count on both sides of its two-pass limit (2,097,152), in row order and
over the clustered copy, 32-bit per-point results (more than 65534 polygons)
with points in more polygons than a result stores.  Radii are zero, mixed
(smaller and larger than an edge-grid cell) and large.  Whole numbers: equal
to the oracle's, bit for bit."""
import functools

import numpy as np
import pytest

import oracle
from paper_2203_14362_gb300 import datagen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402

LIMIT = 4096 * 256


@functools.lru_cache(None)
def case(name):
    mix = g.make_mixture(71)
    rng = np.random.default_rng(71)
    if name == "many":  # 65000 small squares, and 1100 over one place
        x, y = rng.integers(0, (1 << 30) - (1 << 20), (2, 65000))
        lo = np.stack([x, y], 1)
        v = np.concatenate([np.stack([lo, lo + [1 << 20, 0], lo + (1 << 20), lo + [0, 1 << 20]], 1),
                            np.tile(np.array([[0, 0], [1 << 19, 0], [1 << 19, 1 << 19], [0, 1 << 19]])[None], (1100, 1, 1))])
        r = rng.integers(0, 1 << 20, 66100).astype(np.int32)
        pts = g.uniform_points(20_001, 7)
        pts[::40] >>= 9  # in and around the large ones
        return v.reshape(-1, 2).astype(np.int32), np.arange(0, 4 * 66101, 4, dtype=np.uint64), r, pts
    v, o = g.query_polygons(20, 71, mix, vmax=300, r_med=0.02)
    P = o.shape[0] - 1
    r = {"zero": np.zeros(P, np.int32), "mixed": (rng.integers(0, 1 << 12, P) ** 2).astype(np.int32),
         "large": np.full(P, 1 << 25, np.int32)}[name]
    return v, o, r, g.mixture_points(2 * LIMIT + 300, 71, mix)


@pytest.mark.parametrize("name,n,fp32", [("zero", LIMIT + 1, True), ("mixed", LIMIT, True), ("mixed", LIMIT + 1, True),
                                         ("mixed", LIMIT + 1, False), ("large", LIMIT + 1, True), ("many", 20_001, True)])
def test_buffer_join_paths(name, n, fp32):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    v, o, r, pts = case(name)
    pts = pts[:n]
    P = o.shape[0] - 1
    want, want_counts = oracle.buffer_join(pts, v, o, r)
    eng = spx.Engine(0)
    try:
        dpts = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
        ph = eng.load_points(dpts)
        ih = eng.build_buffer_index(eng.load_polygons(v, o), r, fp32_filter=fp32)
        pairs = torch.empty((want.shape[0], 2), dtype=torch.int32, device="cuda")
        counts = torch.full((P,), 7, dtype=torch.int64, device="cuda")
        m = eng.join(ph, ih, pairs, counts)
        assert m == want.shape[0]
        assert np.array_equal(pairs.cpu().numpy().view(np.uint32), want)
        assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
        if P <= 1024:
            ids = torch.empty(m, dtype=torch.int32, device="cuda")
            offs = torch.empty(P + 1, dtype=torch.int64, device="cuda")
            assert eng.select(ph, ih, ids, offs) == m
            order = np.argsort(want[:, 1], kind="stable")
            assert np.array_equal(ids.cpu().numpy().view(np.uint32), want[order, 0])
            assert np.array_equal(offs.cpu().numpy()[1:], np.cumsum(want_counts.astype(np.int64)))
    finally:
        eng.close()


@pytest.mark.parametrize("n", [2 * LIMIT, 2 * LIMIT + 257])
def test_buffer_count_paths(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    v, o, r, pts = case("mixed")
    pts = pts[:n]
    want = oracle.buffer_join(pts, v, o, r)[1]
    eng = spx.Engine(0)
    try:
        dpts = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
        ph = eng.load_points(dpts)
        ih = eng.build_buffer_index(eng.load_polygons(v, o), r)
        counts = torch.full((o.shape[0] - 1,), 7, dtype=torch.int64, device="cuda")
        for table in (ph, eng.cluster_points(ph)):
            counts.fill_(7)
            eng.aggregate(table, ih, counts)
            assert np.array_equal(counts.cpu().numpy().view(np.uint64), want)
    finally:
        eng.close()
