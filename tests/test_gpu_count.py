"""GPU parity of the count aggregate of a table in row order on both sides of
the size where it takes two passes (2,097,152 points), with the block summary
(a coarse map) and without (a fine one), and of counts queued on two streams
at once, which may not share scratch.  Whole numbers: equal to the oracle's."""
import numpy as np
import pytest

import oracle
from paper_2203_14362_gb300 import datagen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402

LIMIT = 1 << 21


@pytest.fixture(scope="module")
def tables():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    mix = g.make_mixture(9)
    pts = g.mixture_points(LIMIT + 300, 9, mix)
    pts[::1001] = -5  # outside the box
    maps = [g.quad_tessellation(20, 15, 9, kmin=2, kmax=60), g.quad_tessellation(130, 120, 9, kmin=2, kmax=6)]
    return pts, maps


@pytest.mark.parametrize("m,fp32", [(0, True), (0, False), (1, True)])
@pytest.mark.parametrize("n", [LIMIT, LIMIT + 1, LIMIT + 257])
def test_count_sizes(tables, m, fp32, n):
    pts, t = tables[0][:n], tables[1][m]
    P = t.ring_off.shape[0] - 1
    _, want = oracle.join_fast(pts, t.verts, t.ring_off)
    eng = spx.Engine(0)
    try:
        dpts = torch.from_numpy(np.ascontiguousarray(pts)).cuda()
        ph = eng.load_points(dpts)
        ih = eng.build_index(eng.load_polygons(t.verts, t.ring_off), fp32_filter=fp32)
        assert eng.index_info(ih)["use_sum"] == (1 if m == 0 else 0)
        counts = torch.full((P,), 3, dtype=torch.int64, device="cuda")
        for _ in range(2):
            eng.aggregate(ph, ih, counts)
            assert np.array_equal(counts.cpu().numpy().view(np.uint64), want)
        g_counts = torch.zeros_like(counts)  # captured, replayed
        graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=s, capture_error_mode="relaxed"):
            eng.aggregate(ph, ih, g_counts)
        for _ in range(2):
            g_counts.fill_(1)
            graph.replay()
            torch.cuda.synchronize()
            assert np.array_equal(g_counts.cpu().numpy().view(np.uint64), want)
    finally:
        eng.close()


def test_two_streams(tables):
    pts, (t, _) = tables
    a, b = pts, np.ascontiguousarray(pts[::-1][: LIMIT + 100])
    eng = spx.Engine(0)
    try:
        ih = eng.build_index(eng.load_polygons(t.verts, t.ring_off))
        P = t.ring_off.shape[0] - 1
        d = [torch.from_numpy(x).cuda() for x in (a, b)]
        want = [oracle.join_fast(x, t.verts, t.ring_off)[1] for x in (a, b)]
        ph = [eng.load_points(x) for x in d]
        out = [[torch.zeros(P, dtype=torch.int64, device="cuda") for _ in range(8)] for _ in range(2)]
        ss = [torch.cuda.Stream(), torch.cuda.Stream()]
        torch.cuda.synchronize()
        for k in range(8):
            for i in range(2):
                eng.aggregate(ph[i], ih, out[i][k], stream=ss[i])
        torch.cuda.synchronize()
        for i in range(2):
            for k in range(8):
                assert np.array_equal(out[i][k].cpu().numpy().view(np.uint64), want[i])
    finally:
        eng.close()
