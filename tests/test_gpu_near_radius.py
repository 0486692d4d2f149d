"""Buffered joins probed where the FP32 distance filter hands over to
the exact test: points around the radius of an edge, within a few units of it, and
beside the perpendiculars through its ends.  Whole numbers: equal to the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2203_14362_gb300 import datagen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402

BOX = 1 << 30


def probes(v, o, r, n, rng):
    q = rng.integers(0, o.shape[0] - 1, n)
    lo, hi = o[q].astype(np.int64), o[q + 1].astype(np.int64)
    i = lo + (rng.random(n) * (hi - lo)).astype(np.int64)
    a, b = v[i].astype(float), v[np.where(i + 1 == hi, lo, i + 1)].astype(float)
    d = b - a
    L = np.maximum(np.sqrt((d * d).sum(1)), 1e-9)
    u = np.where(rng.random(n) < 0.4, rng.integers(0, 2, n), rng.uniform(-0.2, 1.2, n))
    off = r[q] * (1 + rng.normal(0, 1, n) * 10 ** rng.uniform(-12, -2, n)) + rng.integers(-2, 3, n)
    off *= rng.choice([-1.0, 1.0], n)
    p = a + u[:, None] * d + off[:, None] * np.stack([d[:, 1], -d[:, 0]], 1) / L[:, None]
    ang = rng.uniform(0, 2 * np.pi, n)  # around the ends themselves
    p = np.where(rng.random(n)[:, None] < 0.3, a + np.abs(off)[:, None] * np.stack([np.cos(ang), np.sin(ang)], 1), p)
    return np.clip(np.rint(p) + rng.integers(-1, 2, (n, 2)), 0, BOX - 1).astype(np.int32)


@pytest.mark.parametrize("radius", ["small", "mixed", "large"])
@pytest.mark.parametrize("gl", [0, 6])
def test_points_near_the_radius(radius, gl):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(len(radius) + gl)
    v, o = g.query_polygons(24, 9, g.make_mixture(9), vmax=200, r_med=0.03)
    r = {"small": rng.integers(0, 50, 24), "mixed": 10 ** rng.uniform(1, 8, 24), "large": np.full(24, 1 << 26)}[radius].astype(np.int32)
    pts = probes(v, o, r, 150_000, rng)
    want, want_counts = oracle.buffer_join(pts, v, o, r)
    eng = spx.Engine(0)
    try:
        dpts = torch.from_numpy(pts).cuda()
        ph, gh = eng.load_points(dpts), eng.load_polygons(v, o)
        for fp32 in (True, False):
            ih = eng.build_buffer_index(gh, r, grid_log2=gl, fp32_filter=fp32)
            pairs = torch.empty((want.shape[0], 2), dtype=torch.int32, device="cuda")
            counts = torch.zeros(24, dtype=torch.int64, device="cuda")
            assert eng.join(ph, ih, pairs, counts) == want.shape[0]
            assert np.array_equal(pairs.cpu().numpy().view(np.uint32), want)
            assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
    finally:
        eng.close()
