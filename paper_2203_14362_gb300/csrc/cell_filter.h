// FP32 decisions that an exact result backs: which edges a cell's lists keep, and
// the distance test's filter.  Also compiled as plain C++, where their bounds are
// checked against exact integers.
#pragma once

#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define SPX_HD __host__ __device__ __forceinline__
#define SPX_HD_CALL __host__ __device__ __noinline__
#else
#define SPX_HD inline
#define SPX_HD_CALL inline
struct int4 {
    int x, y, z, w;
};
#endif

namespace spx {

// One rounding each, never contracted into a fused multiply-add.  A list is sized
// by one kernel and written by another, both from edge_side or edge_reaches: with
// plain operators the compiler may contract each inlined copy differently, and an
// edge kept by one pass alone would be written past the list.
#ifdef __CUDA_ARCH__
SPX_HD float f_of(int v) { return __int2float_rn(v); }
SPX_HD float f_add(float a, float b) { return __fadd_rn(a, b); }
SPX_HD float f_sub(float a, float b) { return __fsub_rn(a, b); }
SPX_HD float f_mul(float a, float b) { return __fmul_rn(a, b); }
SPX_HD float f_div(float a, float b) { return __fdiv_rn(a, b); }
SPX_HD float f_sqrt(float a) { return __fsqrt_rn(a); }
#else
SPX_HD float f_rounded(float v)
{
    volatile float r = v;
    return r;
}
SPX_HD float f_of(int v) { return static_cast<float>(v); }
SPX_HD float f_add(float a, float b) { return f_rounded(a + b); }
SPX_HD float f_sub(float a, float b) { return f_rounded(a - b); }
SPX_HD float f_mul(float a, float b) { return f_rounded(a * b); }
SPX_HD float f_div(float a, float b) { return f_rounded(a / b); }
SPX_HD float f_sqrt(float a) { return f_rounded(sqrtf(a)); }
#endif

// A cell's points are the integers of [x0, x0 + S) x [y0, y0 + S).
struct CellBox {
    int x0, y0, S;
};

// The part of edge v over the rows of the cell that it straddles, as the cell's
// rightward rays see it: 0 never crossed (left, or no such row), 2 crossed by every
// ray of those rows (right), 1 neither for certain.  An edge whose own x range is
// right of the cell needs no arithmetic.  Else the part's ends come from FP32.  With
// u = 2^-24 and the ends' rows between the edge's: 2 u of |ax| (a conversion and the
// sum) and 6 u of |dx| (two conversions, the division, the rows' conversion, the
// product and the sum), one more u of both in the comparison.  The margin is 2^-18
// = 64 u of |ax| + |dx|, nine times that, and 4 units.
SPX_HD int edge_side(const int4 &v, const CellBox &c)
{
    const int vlo = v.y < v.w ? v.y : v.w, vhi = v.y < v.w ? v.w : v.y;
    const int ylo = c.y0 > vlo ? c.y0 : vlo, yhi = (c.y0 + c.S < vhi ? c.y0 + c.S : vhi) - 1;
    if (ylo > yhi)
        return 0; // straddles no integer row of the cell
    if ((v.x < v.z ? v.x : v.z) >= c.x0 + c.S)
        return 2;
    const float ax = f_of(v.x - c.x0), dx = f_of(v.z - v.x);
    const float slope = f_div(dx, f_of(v.w - v.y));
    const float xa = f_add(ax, f_mul(slope, f_of(ylo - v.y))), xb = f_add(ax, f_mul(slope, f_of(yhi - v.y)));
    const float margin = f_add(4.f, f_mul(3.814697265625e-06f, f_add(fabsf(ax), fabsf(dx)))); // 2^-18
    if (f_sub(fminf(xa, xb), margin) >= f_of(c.S))
        return 2;
    return f_add(fmaxf(xa, xb), margin) < 0.f ? 0 : 1;
}

// May edge v come within r of a point of the cell?  Its distance from the cell's
// centre is compared with r + h + 2, h half the points' diagonal; the rounding of
// the differences (u each, a few of them) is covered by 2^-18 of their sum.
SPX_HD bool edge_reaches(const int4 &v, const CellBox &c, int r)
{
    const float dx = f_of(v.z - v.x), dy = f_of(v.w - v.y), m = f_mul(0.5f, f_of(c.S - 1));
    const float wx = f_add(f_of(c.x0 - v.x), m), wy = f_add(f_of(c.y0 - v.y), m);
    const float dd = f_add(f_mul(dx, dx), f_mul(dy, dy));
    const float t = dd > 0.f ? fminf(1.f, fmaxf(0.f, f_div(f_add(f_mul(wx, dx), f_mul(wy, dy)), dd))) : 0.f;
    const float ex = f_sub(wx, f_mul(t, dx)), ey = f_sub(wy, f_mul(t, dy));
    const float reach = f_add(f_add(f_of(r), f_mul(1.41421366f, m)), 2.f);
    const float sum = f_add(f_add(f_add(fabsf(wx), fabsf(wy)), f_add(fabsf(dx), fabsf(dy))), reach);
    return f_sqrt(f_add(f_mul(ex, ex), f_mul(ey, ey))) <= f_add(reach, f_mul(3.814697265625e-06f, sum)); // 2^-18
}

// Is (px, py) within distance r of the closed segment v = (a, b)?  With
// d = b - a, w = p - a and t = w . d: the distance is |w| when t <= 0, |p - b|
// when t >= |d|^2, else |d x w| / |d|.  Coordinates lie in [0, 2^30], so every
// product of two differences is below 2^60 in magnitude (int64 sums stay
// exact); the last case compares (d x w)^2 with r^2 |d|^2 as 128-bit
// products.  A zero-length edge takes the first case.
SPX_HD_CALL bool seg_near_exact(const int4 &v, int px, int py, int64_t r)
{
    const int64_t dx = (int64_t)v.z - v.x, dy = (int64_t)v.w - v.y;
    const int64_t wx = (int64_t)px - v.x, wy = (int64_t)py - v.y, rr = r * r;
    const int64_t t = wx * dx + wy * dy;
    if (t <= 0)
        return wx * wx + wy * wy <= rr;
    const int64_t dd = dx * dx + dy * dy;
    if (t >= dd) {
        const int64_t ux = (int64_t)px - v.z, uy = (int64_t)py - v.w;
        return ux * ux + uy * uy <= rr;
    }
    const int64_t c = dx * wy - dy * wx;
    const uint64_t ca = (uint64_t)(c < 0 ? -c : c);
#ifdef __CUDA_ARCH__
    const uint64_t lh = __umul64hi(ca, ca), ll = ca * ca;
    const uint64_t rh = __umul64hi((uint64_t)rr, (uint64_t)dd), rl = (uint64_t)rr * (uint64_t)dd;
    return lh < rh || (lh == rh && ll <= rl);
#else
    return (unsigned __int128)ca * ca <= (unsigned __int128)rr * (uint64_t)dd;
#endif
}

// The same with an FP32 filter.  Rounding a coordinate difference costs 2^-24
// relative, so every product of two differences is within 3.01 x 2^-24 of its
// value and a sum or difference of two within 4.1 x 2^-24 of the sum of their
// magnitudes; r |d| (one conversion, half of |d|^2's error, two roundings)
// within 5.2 x 2^-24.  Each comparison trusts FP32 only outside 2^-21 (8 x 2^-24)
// of the magnitudes involved; the rest (near the radius, or near an end's
// perpendicular) is decided exactly.
template <bool FP32>
SPX_HD bool seg_near(const int4 &v, int px, int py, int r)
{
    if (FP32) {
        constexpr float kE = 4.76837158203125e-07f; // 2^-21
        const float dx = f_of(v.z - v.x), dy = f_of(v.w - v.y);
        const float wx = f_of(px - v.x), wy = f_of(py - v.y), rf = f_of(r);
        const float t1 = wx * dx, t2 = wy * dy, t = t1 + t2, et = kE * (fabsf(t1) + fabsf(t2));
        const float dd = dx * dx + dy * dy, rr = rf * rf;
        float a, b, m; // the point is near iff a <= b; m: the magnitudes compared
        bool sure = true;
        if (t < -et) {
            a = wx * wx + wy * wy, b = rr, m = a + b;
        } else if (t - dd > et + kE * dd) {
            const float ux = f_of(px - v.z), uy = f_of(py - v.w);
            a = ux * ux + uy * uy, b = rr, m = a + b;
        } else {
            sure = t > et && dd - t > et + kE * dd;
            const float c1 = dx * wy, c2 = dy * wx;
            a = fabsf(c1 - c2), b = rf * f_sqrt(dd), m = fabsf(c1) + fabsf(c2) + b;
        }
        if (sure && fabsf(a - b) > kE * m)
            return a < b;
    }
    return seg_near_exact(v, px, py, r);
}

} // namespace spx
