"""The FP32 filter of the buffered polygons' distance test, in IEEE float32
(numpy), against exact integers: where it decides, it decides right.  The
points lie around the radius of a segment: at random, within a few units of
it, and beside the perpendiculars through its ends."""
import math

import numpy as np

E = np.float32(2.0 ** -21)


def exact(ax, ay, bx, by, px, py, r):
    dx, dy, wx, wy = bx - ax, by - ay, px - ax, py - ay
    t, dd = wx * dx + wy * dy, dx * dx + dy * dy
    if t <= 0:
        return wx * wx + wy * wy <= r * r
    if t >= dd:
        return (px - bx) ** 2 + (py - by) ** 2 <= r * r
    c = dx * wy - dy * wx
    return c * c <= r * r * dd


def filtered(ax, ay, bx, by, px, py, r):
    """True / False, or None where the filter leaves it to the exact test."""
    f = np.float32
    dx, dy, wx, wy, rf = f(bx - ax), f(by - ay), f(px - ax), f(py - ay), f(r)
    t1, t2 = wx * dx, wy * dy
    t, et = t1 + t2, E * (abs(t1) + abs(t2))
    dd, rr = dx * dx + dy * dy, rf * rf
    if t < -et:
        a, b = wx * wx + wy * wy, rr
        m = a + b
    elif t - dd > et + E * dd:
        ux, uy = f(px - bx), f(py - by)
        a, b = ux * ux + uy * uy, rr
        m = a + b
    else:
        if not (t > et and dd - t > et + E * dd):
            return None
        c1, c2 = dx * wy, dy * wx
        a, b = abs(c1 - c2), rf * np.sqrt(dd)
        m = abs(c1) + abs(c2) + b
    return bool(a < b) if abs(a - b) > E * m else None


def test_filter_never_wrong():
    rng = np.random.default_rng(3)
    B = 1 << 30
    decided = near = 0
    for k in range(30000):
        scale = 10 ** rng.uniform(0, 9)
        ax, ay = (int(v) for v in rng.integers(0, B, 2))
        bx = int(min(max(ax + rng.normal() * scale, 0), B))
        by = int(min(max(ay + rng.normal() * scale, 0), B))
        r = int(min(10 ** rng.uniform(0, 9), B - 1))
        L = math.hypot(bx - ax, by - ay)
        u = rng.uniform(-0.2, 1.2) if k % 3 else float(rng.integers(0, 2))  # along the segment; at its ends
        off = r * (1 + rng.normal() * 10 ** rng.uniform(-12, 0)) + rng.integers(-2, 3)
        nx, ny = ((by - ay) / L, -(bx - ax) / L) if L else (1.0, 0.0)
        px = int(min(max(ax + u * (bx - ax) + off * nx, 0), B - 1))
        py = int(min(max(ay + u * (by - ay) + off * ny, 0), B - 1))
        got = filtered(ax, ay, bx, by, px, py, r)
        if got is not None:
            decided += 1
            assert got == exact(ax, ay, bx, by, px, py, r), (ax, ay, bx, by, px, py, r)
        else:
            near += 1
    assert decided > 10000 and near > 500
