"""The ctx's pool under memory pressure: what it keeps between calls is there for the
calls that allocate from the device."""
import numpy as np
import pytest

from paper_2203_14362_gb300 import datagen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402

MB = 1 << 20


@pytest.fixture()
def eng():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    e = spx.Engine(0)
    yield e
    e.close()


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_buffered_build_keeps_only_the_index(eng):
    # 256 queries of many vertices: the local lists' temporaries are larger than what
    # the pool's blocks round up to
    mix = g.make_mixture(3)
    v, o = g.query_polygons(8, 3, mix, vmax=300, r_med=0.05)
    eng.free(eng.build_buffer_index(eng.load_polygons(v, o), np.zeros(8, np.int32)))  # kernels loaded
    v, o = g.query_polygons(256, 3, mix, vmax=5000, r_med=0.02)
    gh = eng.load_polygons(v, o)
    before = free_bytes()
    ih = eng.build_buffer_index(gh, np.full(256, 1 << 18, np.int32), grid_log2=9)
    held, own = before - free_bytes(), eng.index_info(ih)["device_bytes"]
    assert held <= own + 64 * MB


def test_scratch_freed_on_another_stream(eng):
    # a count's scratch (32 MB) is still in use on a caller's stream when a table needs
    # memory that is only there once that scratch goes back
    n = 1 << 28
    t = g.quad_tessellation(16, 16, 5, kmin=4, kmax=20)
    ih = eng.build_index(eng.load_polygons(t.verts, t.ring_off), grid_log2=8)
    pts = torch.zeros((n, 2), dtype=torch.int32, device="cuda")
    ph = eng.load_points(pts)
    counts = torch.zeros(256, dtype=torch.int64, device="cuda")
    eng.aggregate(ph, ih, counts)
    want = counts.clone()
    table = np.zeros((7 * MB, 2), np.int32)  # 56 MB
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(1000)
    hog = torch.empty(free_bytes() - 40 * MB, dtype=torch.uint8, device="cuda")
    try:
        with torch.cuda.stream(s):
            torch.cuda._sleep(1_000_000_000)  # about half a second
            eng.aggregate(ph, ih, counts, stream=s)
        few = eng.load_points(table)
        torch.cuda.synchronize()
        assert torch.equal(counts, want)
        eng.aggregate(few, ih, counts)
        assert counts.sum().item() == (7 * MB if want.sum().item() else 0)
        assert eng.points_info(few)["n"] == 7 * MB
    finally:
        del hog
        torch.cuda.empty_cache()


def test_freed_table_gives_back_the_pool(eng):
    t = g.quad_tessellation(30, 30, 7, kmin=4, kmax=100)
    gh = eng.load_polygons(t.verts, t.ring_off)
    few = np.zeros((1000, 2), np.int32)
    eng.free(eng.build_index(gh, grid_log2=6, on_device=True))  # kernels loaded
    eng.free(eng.load_points(few))
    before = free_bytes()
    eng.free(eng.build_index(gh, grid_log2=12, on_device=True))
    assert free_bytes() < before - 256 * MB  # kept for the next build
    eng.free(eng.load_points(few))
    assert free_bytes() >= before - 8 * MB
