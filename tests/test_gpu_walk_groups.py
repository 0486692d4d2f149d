"""GPU parity where pass 1b shares its rows out in groups of fewer than 32 bitmap words:
counts over clustered tables from one point to several million, whose directory
leaves runs of marked rows, and joins with 32-bit results (more than 65534 polygons).
Whole numbers: equal to the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2203_14362_gb300 import datagen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402

BOX = 1 << 30


@pytest.fixture(scope="module")
def eng():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    e = spx.Engine(0)
    yield e
    e.close()


def overlapping(k):  # k star polygons over one place
    rng = np.random.default_rng(k)
    th = np.linspace(0, 2 * np.pi, 30, endpoint=False)
    r = (1 << 27) * rng.uniform(0.3, 1.0, (k, 30))
    c = BOX // 2 + rng.integers(-(1 << 25), 1 << 25, (k, 2))
    v = np.stack([c[:, :1] + r * np.cos(th), c[:, 1:] + r * np.sin(th)], 2).reshape(-1, 2)
    return np.clip(v, 0, BOX).astype(np.int32), np.arange(0, 30 * k + 1, 30, dtype=np.uint64)


@pytest.mark.parametrize("n,k", [(1, 25), (31, 25), (33, 25), (257, 2100), (40_000, 25), (20_000, 2100), (311_111, 25),
                                 (1_300_003, 3), (5_200_001, 3)])
def test_clustered_counts(eng, n, k):
    v, o = overlapping(k)
    pts = g.uniform_points(n, n)
    pts[::3] = BOX // 2 + (pts[::3] >> 4) - (1 << 25)
    pts[::501] = -1
    want = oracle.join_fast(pts, v, o)[1]
    dpts = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
    ch = eng.cluster_points(eng.load_points(dpts))
    gh = eng.load_polygons(v, o)
    for gl in (5, 9 if k < 100 else 6):
        ih = eng.build_index(gh, grid_log2=gl)
        counts = torch.full((k,), 7, dtype=torch.int64, device="cuda")
        eng.stats(reset=True)
        eng.aggregate(ch, ih, counts)
        assert np.array_equal(counts.cpu().numpy().view(np.uint64), want)
        assert eng.stats()["points_scanned"] == n  # marked rows and those of the directory, once each
        eng.free(ih)


@pytest.mark.parametrize("n", [33_000, 1_100_003])
def test_wide_joins(eng, n):
    rng = np.random.default_rng(3)
    lo = rng.integers(0, BOX - (1 << 21), (66_000, 2))
    s = 1 << 21
    v = np.stack([lo, lo + [s, 0], lo + s, lo + [0, s]], 1).reshape(-1, 2).astype(np.int32)
    o = np.arange(0, 4 * 66_001, 4, dtype=np.uint64)
    pts = g.uniform_points(n, 9)
    want, want_counts = oracle.join_fast(pts, v, o)
    dpts = torch.from_numpy(pts).cuda()
    ph = eng.load_points(dpts)
    ih = eng.build_index(eng.load_polygons(v, o), grid_log2=10)
    pairs = torch.empty((want.shape[0], 2), dtype=torch.int32, device="cuda")
    counts = torch.zeros(66_000, dtype=torch.int64, device="cuda")
    assert eng.join(ph, ih, pairs, counts) == want.shape[0]
    assert np.array_equal(pairs.cpu().numpy().view(np.uint32), want)
    assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
