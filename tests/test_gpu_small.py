"""GPU parity of the join on both sides of the small-table limit (1,048,576
points): the two-launch path (one pass-1 kernel, offsets summed in the emit
kernel) and the split passes, at chunk and CTA edges, with counts in shared
and in global memory, 16-bit and 32-bit per-point results.  Pairs, counts and
totals are whole numbers: equal to the oracle's, bit for bit."""
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
def polygons(kind):
    if kind == "tess":  # 2500 cells: more than the small path counts in shared memory
        t = g.quad_tessellation(50, 50, 3, kmin=2, kmax=20)
        return t.verts, t.ring_off
    if kind == "squares":  # 65536 overlapping squares: 32-bit results, points in up to four
        s = (1 << 30) // 256
        x, y = np.meshgrid(np.arange(256), np.arange(256))
        lo = np.stack([x.ravel() * s, y.ravel() * s], 1)
        hi = np.minimum(lo + s + s // 3, 1 << 30)
        v = np.stack([lo, np.stack([hi[:, 0], lo[:, 1]], 1), hi, np.stack([lo[:, 0], hi[:, 1]], 1)], 1)
        return v.reshape(-1, 2).astype(np.int32), np.arange(0, 4 * 65537, 4, dtype=np.uint64)
    mix = g.make_mixture(5)
    return g.query_polygons(40, 5, mix, vmax=600, r_med=0.03)


@pytest.mark.parametrize("kind", ["tess", "squares", "queries"])
@pytest.mark.parametrize("n,fp32", [(1, True), (255, False), (257, True), (2048, True), (2049, False), (LIMIT, True),
                                    (LIMIT + 1, True), (LIMIT + 1, False)])
def test_join_sizes(kind, n, fp32):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    v, o = polygons(kind)
    P = o.shape[0] - 1
    pts = g.uniform_points(n, n)
    want, want_counts = oracle.join_fast(pts, v, o)
    eng = spx.Engine(0)
    try:
        dpts = torch.from_numpy(pts).cuda()
        ph = eng.load_points(dpts)
        ih = eng.build_index(eng.load_polygons(v, o), grid_log2=9, fp32_filter=fp32)
        pairs = torch.empty((max(want.shape[0], 1), 2), dtype=torch.int32, device="cuda")
        counts = torch.full((P,), 7, dtype=torch.int64, device="cuda")
        total = torch.zeros(1, dtype=torch.int64, device="cuda")
        for t in (None, total):  # the library's own total word, the caller's
            m = eng.join(ph, ih, pairs, counts, t)
            assert m == want.shape[0] and (t is None or int(t) == m)
            assert np.array_equal(pairs[:m].cpu().numpy().view(np.uint32), want)
            assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
        if m > 1:  # too little room: the size that is needed, and the pairs that fit
            with pytest.raises(spx.SpxError) as e:
                eng.join(ph, ih, pairs[:m - 1], counts)
            assert e.value.status == spx.SPX_ECAPACITY and str(m) in str(e.value)
            assert np.array_equal(pairs[:m - 1].cpu().numpy().view(np.uint32), want[:m - 1])
            with pytest.raises(spx.SpxError):
                eng.join(ph, ih, None, counts)  # sizing call without an output
            assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
    finally:
        eng.close()
