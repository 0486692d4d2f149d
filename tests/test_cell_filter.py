"""The FP32 decisions behind the edge lists and the distance filter, as the source
has them (csrc/cell_filter.h compiled as C++), against exact integers, at sizes
around each decision's line.  The two that size lists in one kernel and write them
in another decide alike however the compiler contracts products and sums."""
import ctypes
import os
import platform
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2203_14362_gb300", "csrc")
BOX = 1 << 30
DRIVER = r"""
#include "cell_filter.h"
using namespace spx;
extern "C" void sides(int n, const int4 *v, const CellBox *c, int *out) { for (int i = 0; i < n; ++i) out[i] = edge_side(v[i], c[i]); }
extern "C" void reaches(int n, const int4 *v, const CellBox *c, const int *r, int *out)
{ for (int i = 0; i < n; ++i) out[i] = edge_reaches(v[i], c[i], r[i]); }
extern "C" void nears(int n, const int4 *v, const int *p, const int *r, int *fast, int *exact)
{ for (int i = 0; i < n; ++i) { fast[i] = seg_near<true>(v[i], p[2 * i], p[2 * i + 1], r[i]);
                                exact[i] = seg_near<false>(v[i], p[2 * i], p[2 * i + 1], r[i]); } }
"""


def has_fma():
    if platform.machine() == "aarch64":
        return True
    try:
        return " fma " in open("/proc/cpuinfo").read()
    except OSError:
        return False


@pytest.fixture(scope="module")
def libs(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("cell_filter")
    (d / "driver.cpp").write_text(DRIVER)
    out = []
    fma = [] if platform.machine() == "aarch64" else ["-mfma"]
    for name, flags in [("off", ["-ffp-contract=off"])] + ([("fast", ["-ffp-contract=fast", *fma])] if has_fma() else []):
        so = str(d / f"{name}.so")
        subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", *flags, "-I", CSRC, "-o", so, str(d / "driver.cpp")],
                       check=True)
        out.append(ctypes.CDLL(so))
    return out


def call(fn, n, *arrays):
    fn(ctypes.c_int(n), *[a.ctypes.data_as(ctypes.c_void_p) for a in arrays])


def ints(*cols):
    return np.ascontiguousarray(np.stack(cols, 1).astype(np.int32))


def crosses(v, px, py):
    """The exact crossing rule, on Python integers (object arrays)."""
    ax, ay, bx, by = v
    d = (bx - ax) * (py - ay) - (by - ay) * (px - ax)
    return ((ay > py) != (by > py)) & (d != 0) & ((d > 0) == (by > ay))


def test_edge_side(libs):
    rng = np.random.default_rng(1)
    n = 400_000
    a, b = rng.integers(0, BOX + 1, (2, n, 2))
    short = rng.random(n) < 0.5  # edges of any length
    step = (rng.normal(0, 1, (n, 2)) * 2.0 ** rng.uniform(2, 28, (n, 1))).astype(np.int64)
    b = np.where(short[:, None], np.clip(a + step, 0, BOX), b)
    S = 1 << rng.integers(14, 28, n)
    y0 = np.clip((a[:, 1] + rng.random(n) * (b[:, 1] - a[:, 1]) - rng.random(n) * S).astype(np.int64), 0, BOX - S)
    # the cell's right or left border beside the edge's part over its rows, within the margin's size or at random
    ylo = np.maximum(y0, np.minimum(a[:, 1], b[:, 1]))
    yhi = np.minimum(y0 + S, np.maximum(a[:, 1], b[:, 1])) - 1
    dy = np.where(a[:, 1] == b[:, 1], 1, b[:, 1] - a[:, 1])
    at = a[:, 0] + (np.where(rng.random(n) < 0.5, ylo, yhi) - a[:, 1]) / dy * (b[:, 0] - a[:, 0])
    margin = 4 + 2.0 ** -18 * (np.abs(a[:, 0] - at) + np.abs(b[:, 0] - a[:, 0]) + S)
    off = rng.uniform(-2, 2, n) * margin
    x0 = np.clip(np.where(rng.random(n) < 0.5, at - S - off, at + off), 0, BOX - S).astype(np.int64)
    v, c = ints(a[:, 0], a[:, 1], b[:, 0], b[:, 1]), ints(x0, y0, S)
    got = [np.empty(n, np.int32) for _ in libs]
    for lib, g in zip(libs, got):
        call(lib.sides, n, v, c, g)
        assert np.array_equal(g, got[0])  # one decision, whatever is contracted
    side = got[0]
    rows = ylo <= yhi
    obj = [x.astype(object) for x in (a[:, 0], a[:, 1], b[:, 0], b[:, 1])]
    for y in (ylo, yhi):  # the crossing's x is monotone over the rows: both ends decide them all
        right = crosses(obj, (x0 + S - 1).astype(object), y.astype(object)).astype(bool)
        left = crosses(obj, x0.astype(object), y.astype(object)).astype(bool)
        assert right[rows & (side == 2)].all()
        assert not left[rows & (side == 0)].any()
    assert (side[~rows] == 0).all()
    assert min((side[rows] == k).sum() for k in range(3)) > 10_000


def test_edge_reaches(libs):
    rng = np.random.default_rng(2)
    n = 400_000
    a = rng.integers(0, BOX + 1, (n, 2))
    b = np.clip(a + (rng.normal(0, 1, (n, 2)) * 2.0 ** rng.uniform(0, 30, (n, 1))).astype(np.int64), 0, BOX)
    S = 1 << rng.integers(0, 26, n)
    x0, y0 = (np.clip(a + (rng.normal(0, 1, (n, 2)) * 2.0 ** rng.uniform(4, 30, (n, 1))).astype(np.int64), 0, BOX - S[:, None])).T
    # radii around the one at which the cell's nearest corner or centre is just reached
    d, w = (b - a).astype(float), np.stack([x0, y0], 1) + (S - 1)[:, None] / 2 - a
    dd = np.maximum((d * d).sum(1), 1)
    t = np.clip((w * d).sum(1) / dd, 0, 1)[:, None]
    dist = np.sqrt(((w - t * d) ** 2).sum(1))
    k = rng.integers(0, 3, n)
    r = np.where(k == 0, dist - 0.70710678 * (S - 1) - 2, np.where(k == 1, dist - (S - 1) / 2, dist))
    r = np.clip(r * (1 + rng.normal(0, 1, n) * 2.0 ** -20) + rng.integers(-3, 4, n), 0, BOX - 1).astype(np.int64)
    v, c, ri = ints(a[:, 0], a[:, 1], b[:, 0], b[:, 1]), ints(x0, y0, S), np.ascontiguousarray(r.astype(np.int32))
    got = [np.empty(n, np.int32) for _ in libs]
    for lib, g in zip(libs, got):
        call(lib.reaches, n, v, c, ri, g)
        assert np.array_equal(g, got[0])
    # an edge left out comes within r of none of the cell's points: its corners, the
    # points nearest the edge's ends, and random ones
    fast, exact = np.empty(n, np.int32), np.empty(n, np.int32)
    probes = [(x0, y0), (x0 + S - 1, y0), (x0, y0 + S - 1), (x0 + S - 1, y0 + S - 1)]
    probes += [(np.clip(e[:, 0], x0, x0 + S - 1), np.clip(e[:, 1], y0, y0 + S - 1)) for e in (a, b, (a + t * d).astype(np.int64))]
    probes += [(x0 + (rng.random(n) * S).astype(np.int64), y0 + (rng.random(n) * S).astype(np.int64)) for _ in range(4)]
    for px, py in probes:
        call(libs[0].nears, n, v, ints(np.minimum(px, BOX - 1), np.minimum(py, BOX - 1)), ri, fast, exact)
        assert not exact[got[0] == 0].any()
    assert 10_000 < (got[0] == 0).sum() < n - 10_000


def test_seg_near(libs):
    rng = np.random.default_rng(3)
    n = 600_000
    a = rng.integers(0, BOX + 1, (n, 2))
    b = np.clip(a + (rng.normal(0, 1, (n, 2)) * 10 ** rng.uniform(0, 9, (n, 1))).astype(np.int64), 0, BOX)
    r = np.minimum(10 ** rng.uniform(0, 9, n), BOX - 1).astype(np.int64)
    d = (b - a).astype(float)
    L = np.maximum(np.sqrt((d * d).sum(1)), 1e-9)
    u = np.where(rng.random(n) < 1 / 3, rng.integers(0, 2, n), rng.uniform(-0.2, 1.2, n))  # beside the ends' perpendiculars
    off = r * (1 + rng.normal(0, 1, n) * 10 ** rng.uniform(-12, 0, n)) + rng.integers(-2, 3, n)
    p = a + u[:, None] * d + off[:, None] * np.stack([d[:, 1], -d[:, 0]], 1) / L[:, None]
    p = ints(*np.clip(np.rint(p), 0, BOX - 1).T)
    v, ri = ints(a[:, 0], a[:, 1], b[:, 0], b[:, 1]), np.ascontiguousarray(r.astype(np.int32))
    fast, exact = np.empty(n, np.int32), np.empty(n, np.int32)
    for lib in libs:
        call(lib.nears, n, v, p, ri, fast, exact)
        assert np.array_equal(fast, exact)
    # the exact test itself, on Python integers
    for i in rng.integers(0, n, 4000):
        (ax, ay), (bx, by), (px, py), rr = map(int, a[i]), map(int, b[i]), map(int, p[i]), int(r[i]) ** 2
        dx, dy, wx, wy = bx - ax, by - ay, px - ax, py - ay
        t, dd = wx * dx + wy * dy, dx * dx + dy * dy
        near = (wx * wx + wy * wy <= rr if t <= 0 else (px - bx) ** 2 + (py - by) ** 2 <= rr if t >= dd
                else (dx * wy - dy * wx) ** 2 <= rr * dd)
        assert near == bool(exact[i])
    assert 100_000 < exact.sum() < n - 100_000
