"""The polygon indexes whose cells list many edges do hold local lists: their device
memory exceeds that of the arrays they were built from.  And a tuner's limit on an
index's bytes covers those lists."""
import numpy as np
import pytest

import oracle
from paper_2203_14362_gb300 import datagen as g
from test_gpu_local_lists import rings

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402

BOUNDARY = 1


def array_bytes(host, gl):
    """What the index takes without local lists: its arrays, the cover bitmap and the
    block summary, each a multiple of 256 bytes."""
    sizes = [host[k].nbytes for k in ("coarse", "fine", "entries", "edges")]
    sizes += [max(4 ** min(gl, 8) // 8, 4), max(2 * 4 ** min(gl, 8), 16)]
    return sum((s + 255) // 256 * 256 for s in sizes) + 256


@pytest.fixture(scope="module")
def eng():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    e = spx.Engine(0)
    yield e
    e.close()


@pytest.mark.parametrize("name", ["tess", "spikes", "scribble", "lattice"])
@pytest.mark.parametrize("gl,sub", [(3, 1), (5, 3), (7, 2), (8, 3)])
def test_lists_are_there(eng, name, gl, sub):
    v, o = rings(name, np.random.default_rng(len(name) * 100 + gl))  # those of test_local_lists
    host = spx.host_index(v, o, gl, sub)
    ent = host["entries"].reshape(-1, 4)
    z = ent[(ent[:, 3] & BOUNDARY) != 0, 2]
    long_lists = z.mean() >= 8 and z.max() >= 8
    gh = eng.load_polygons(v, o)
    for on_device in (False, True):
        ih = eng.build_index(gh, grid_log2=gl, sub_log2=sub, on_device=on_device)
        own = eng.index_info(ih)["device_bytes"]
        assert own > array_bytes(host, gl) if long_lists else own == array_bytes(host, gl)
        eng.free(ih)
    assert long_lists or name in ("tess", "scribble")  # both sides of the rule are among the cases


def test_tuner_limit_covers_local_lists(eng):
    v, o = rings("spikes", np.random.default_rng(605))
    pts = g.uniform_points(100_000, 6)
    counts = oracle.join_fast(pts, v, o)[1]
    dpts = torch.from_numpy(pts).cuda()
    ph, gh = eng.load_points(dpts), eng.load_polygons(v, o)
    with_lists = eng.index_info(eng.build_index(gh, grid_log2=5, sub_log2=3))["device_bytes"]
    plain = array_bytes(spx.host_index(v, o, 5, 3), 5)
    assert plain < with_lists
    for limit in (plain, with_lists - 1, with_lists):
        _, trials, ih = eng.autotune(ph, gh, grid_min=5, grid_max=5, reps=1, max_index_bytes=limit)
        assert all(t["device_bytes"] <= limit for t in trials)
        assert {t["sub_log2"]: t["device_bytes"] for t in trials}[3] == (with_lists if limit == with_lists else plain)
        got = torch.zeros(o.shape[0] - 1, dtype=torch.int64, device="cuda")
        eng.aggregate(ph, ih, got)
        assert np.array_equal(got.cpu().numpy().view(np.uint64), counts)
