"""Distance queries where the device has no memory for the packed ids (8 B per point,
which they can do without): the answers are the same, calls of the same size neither
take nor give back device memory, and a captured join replays right after them."""
import numpy as np
import pytest

from paper_2203_14362_gb300 import datagen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402

N = 16_000_000  # packed ids: 128 MB; the other scratch: about 100 MB


def test_no_room_for_packed_ids():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    mix = g.make_mixture(5)
    v, o = g.query_polygons(12, 5, mix, vmax=60, r_med=0.01)
    r = np.full(12, 1 << 21, np.int32)
    dpts = torch.from_numpy(np.ascontiguousarray(g.mixture_points(N, 5, mix))).cuda()
    P = 12

    def calls(eng, ph, ih, pairs, ids, offs):
        counts = torch.zeros(P, dtype=torch.int64, device="cuda")
        m = eng.select(ph, ih, ids, offs)
        assert eng.join(ph, ih, pairs, counts) == m
        return m, counts

    eng = spx.Engine(0)
    try:  # with room: what is expected
        pairs, ids = (torch.zeros(s, dtype=torch.int32, device="cuda") for s in ((4_000_000, 2), (4_000_000,)))
        offs = torch.zeros(P + 1, dtype=torch.int64, device="cuda")
        m, counts = calls(eng, eng.load_points(dpts), eng.build_buffer_index(eng.load_polygons(v, o), r), pairs, ids, offs)
        want = [t[:m].clone() for t in (pairs, ids)] + [offs.clone(), counts.clone()]
    finally:
        eng.close()
    eng = spx.Engine(0)
    hog = None
    try:
        ph = eng.load_points(dpts)
        ih = eng.build_buffer_index(eng.load_polygons(v, o), r)
        few = eng.load_points(dpts[:1_200_000].clone())
        calls(eng, few, ih, pairs, ids, offs)  # the kernels are loaded
        total = torch.zeros(1, dtype=torch.int64, device="cuda")
        got_counts = torch.zeros(P, dtype=torch.int64, device="cuda")
        s = torch.cuda.Stream()
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        hog = torch.empty(torch.cuda.mem_get_info()[0] - (180 << 20), dtype=torch.uint8, device="cuda")
        for k in range(4):
            if k == 1:
                with torch.cuda.graph(graph, stream=s, capture_error_mode="relaxed"):
                    eng.join(ph, ih, pairs, got_counts, total=total, sync=False, stream=s)
            pairs.zero_()
            ids.zero_()
            m2, counts = calls(eng, ph, ih, pairs, ids, offs)
            assert m2 == m
            for a, b in zip((pairs[:m], ids[:m], offs, counts), want):
                assert torch.equal(a, b)
            if k < 2:  # the comparisons and the capture have taken what they need
                free = torch.cuda.mem_get_info()[0]
                assert free < N * 8  # the ids did not fit beside the scratch
            assert torch.cuda.mem_get_info()[0] == free
        pairs.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert total.item() == m and torch.equal(pairs[:m], want[0]) and torch.equal(got_counts, want[3])
    finally:
        del hog
        torch.cuda.empty_cache()
        eng.close()
