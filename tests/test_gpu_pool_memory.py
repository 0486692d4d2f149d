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
