"""Host tables and host-built indexes used at once on a stream that does not wait
for the legacy stream: the upload is on the device when the call returns.  Sizes
below, at and above the driver's staging buffer; a fresh engine each time, so that
the memory held other bytes before.  (A wait that is missing shows by chance
only; what these cases pin is the order of upload, local lists, join and clustering.)"""
import numpy as np
import pytest

import oracle
from paper_2203_14362_gb300 import datagen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402


@pytest.mark.parametrize("n", [1001, 8192, 8193, 700_001])
def test_upload_then_other_stream(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    mix = g.make_mixture(n)
    v, o = g.query_polygons(12, n, mix, vmax=900, r_med=0.05)  # long lists on a coarse grid
    pts = g.mixture_points(n, n, mix)
    want, want_counts = oracle.join_fast(pts, v, o)
    s = torch.cuda.Stream()
    for _ in range(3):
        eng = spx.Engine(0)
        try:
            pairs = torch.empty((max(want.shape[0], 1), 2), dtype=torch.int32, device="cuda")
            counts = torch.zeros(o.shape[0] - 1, dtype=torch.int64, device="cuda")
            torch.cuda.synchronize()
            with torch.cuda.stream(s):
                ph = eng.load_points(pts)
                ih = eng.build_index(eng.load_polygons(v, o), grid_log2=5)
                m = eng.join(ph, ih, pairs, counts, stream=s)
                assert m == want.shape[0]
                assert np.array_equal(pairs[:m].cpu().numpy().view(np.uint32), want)
                assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
                ch = eng.cluster_points(eng.load_points(pts))
                counts.fill_(1)
                eng.aggregate(ch, ih, counts, stream=s)
                s.synchronize()
                assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
        finally:
            eng.close()
