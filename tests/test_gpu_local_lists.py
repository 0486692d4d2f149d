"""GPU parity of the exact tests through local edge lists: polygon indexes whose
cells list many edges (coarse grids, many vertices, spikes that reach across the
box, self-intersections, vertices on and beside cell borders), probed at random,
on and beside vertices, and along cell borders.  Pairs and counts equal the
oracle's, bit for bit; the index's arrays stay the host build's, byte for byte,
although the lists replace what the kernels read."""
import numpy as np
import pytest

import oracle
from paper_2203_14362_gb300 import datagen as g

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2203_14362_gb300 import spx  # noqa: E402

BOX = 1 << 30


def rings(name, rng):
    if name == "tess":
        t = g.quad_tessellation(7, 6, 5, kmin=40, kmax=400)
        return t.verts, t.ring_off
    parts = []
    for k in range(14):
        m = int(rng.integers(40, 400))
        if name == "spikes":  # long thin teeth across the box, every other vertex far away
            x = np.sort(rng.integers(0, BOX, m))
            y = np.where(np.arange(m) % 2, rng.integers(0, BOX, m), rng.integers(0, BOX >> 4, m))
            p = np.stack([x, y], 1) if k % 2 else np.stack([y, x], 1)
        elif name == "scribble":  # self-intersecting, many short edges in few cells
            c = rng.integers(BOX // 4, 3 * BOX // 4, 2)
            p = np.clip(c + np.cumsum(rng.normal(0, 1 << 22, (m, 2)), 0), 0, BOX)
        else:  # vertices on and one unit beside the borders of cells of 2^22 units, horizontal edges among them
            p = (rng.integers(100, 140, (m, 2)) << 22) + rng.integers(-1, 2, (m, 2))
            p[::5, 1] = p[1::5, 1][: len(p[::5])] if m % 5 == 0 else p[::5, 1]
        parts.append(p.astype(np.int64))
    v = np.concatenate(parts).astype(np.int32)
    o = np.zeros(len(parts) + 1, np.uint64)
    o[1:] = np.cumsum([len(p) for p in parts])
    return v, o


@pytest.mark.parametrize("name", ["tess", "spikes", "scribble", "lattice"])
@pytest.mark.parametrize("gl,sub,fp32", [(3, 1, True), (5, 3, True), (7, 2, False), (8, 3, True)])
def test_local_lists(name, gl, sub, fp32):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(len(name) * 100 + gl)
    v, o = rings(name, rng)
    near = v[rng.integers(0, v.shape[0], 40_000)].astype(np.int64) + rng.integers(-2, 3, (40_000, 2))
    side = 1 << (30 - gl - sub)
    border = near // side * side + rng.integers(-1, 2, near.shape)
    spread = v[rng.integers(0, v.shape[0], 40_000)] + rng.normal(0, 1 << 23, (40_000, 2)).astype(np.int64)
    pts = np.concatenate([g.uniform_points(60_000, gl), near, border, spread])
    pts = np.clip(pts, 0, BOX - 1).astype(np.int32)
    want, want_counts = oracle.join_fast(pts, v, o)
    eng = spx.Engine(0)
    try:
        gh = eng.load_polygons(v, o)
        dpts = torch.from_numpy(pts).cuda()
        ph = eng.load_points(dpts)
        pairs = torch.empty((want.shape[0], 2), dtype=torch.int32, device="cuda")
        counts = torch.zeros(o.shape[0] - 1, dtype=torch.int64, device="cuda")
        host = spx.host_index(v, o, gl, sub)
        for on_device in (False, True):
            ih = eng.build_index(gh, grid_log2=gl, sub_log2=sub, fp32_filter=fp32, on_device=on_device)
            got = eng.index_arrays(ih)
            for k in ("coarse", "fine", "entries", "edges"):
                assert np.array_equal(got[k].ravel(), host[k].ravel()), k
            for plain in (False, True):
                m = eng.join(ph, ih, pairs, counts, plain=plain)
                assert m == want.shape[0]
                assert np.array_equal(pairs.cpu().numpy().view(np.uint32), want)
                assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
            counts.fill_(1)
            eng.aggregate(ph, ih, counts)
            assert np.array_equal(counts.cpu().numpy().view(np.uint64), want_counts)
            eng.free(ih)
    finally:
        eng.close()
