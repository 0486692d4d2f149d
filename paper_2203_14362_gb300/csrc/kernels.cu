// sm_103a kernels of libspx: the point-in-polygon join, count aggregate and
// the plain comparison join (SPADE §5.2 selection / join / aggregation: the
// per-point work of the paper's fragment shader -- mask with exact boundary
// tests, additive blend for counts, Map with scan compaction, §5.1).
//
// Per point:
//   coarse word  (y >> sc) << g | (x >> sc)      -- geometric transform to a cell
//   mixed cell   -> fine word of the cell's F x F block
//   resolved word: none / one INSIDE polygon / entry list
//   entry INSIDE -> the point is in the polygon       -- mask, inside pixel
//         BOUNDARY -> crossing parity over the fine row's edges  -- boundary pixel
// The crossing rule is exact: an edge a->b counts iff it straddles y
// ((a.y > y) != (b.y > y)) and the orientation d = (b.x-a.x)(y-a.y) -
// (b.y-a.y)(x-a.x) is nonzero with the sign of b.y - a.y.  The sign of d comes
// from FP32 when |d_f| > 2^-21 (|t1| + |t2|) (forward error bound of the FP32
// evaluation with a factor-2 margin), else from an exact int64 recomputation.
//
// The join is a cached two-pass Map (§5.1), the same for polygons, buffered
// polygons and disks.  Pass 1a (k_resolve_sum; k_resolve without the block
// summary) is persistent and barrier-free: every warp takes its own 256-point
// chunks, resolves their cells, stores a result per point (2 bytes up to 65534
// polygons, else 4) and marks the rows whose cell holds an entry list; pass 1b
// (k_walk) walks those lists 32 rows at a time.  A device-wide scan turns the
// chunks' pair totals into offsets, and pass 3 (k_wemit16; k_wemit for 4-byte
// results) writes each chunk's pairs in point order.  Small tables take one
// pass-1 kernel (k_small), and so do many disks (k_disk_pass1).  The count aggregate
// is pass 1 alone, or k_warp.
// Serving batches (k_multi) and the selection partition (k_part_*) follow.
#include "cell_filter.h"
#include "kernels.h"
#include "spx_internal.h"

#include <algorithm>
#include <climits>
#include <type_traits>
#include <cuda_runtime.h>

namespace spx {
namespace {

#ifndef SPX_TILE_THREADS
#define SPX_TILE_THREADS 256
#endif
constexpr int kThreads = SPX_TILE_THREADS;  // threads per CTA of the persistent kernels
constexpr int kWarps = kThreads / 32;
constexpr int kPlainThreads = 256;          // threads per CTA of the plain kernels
constexpr uint32_t kFull = 0xffffffffu;
// Pass-1 result of a point (4 bytes):
//   kResNone                            in no polygon
//   q (bit 31 clear)                    in exactly polygon q
//   kResMulti | kResCount | c<<20 | q   in c polygons (2 <= c <= 1022), the first q < 2^20
//   kResMulti | q                       in several polygons, the first q (count not stored)
constexpr uint32_t kResNone = 0xffffffffu;
constexpr uint32_t kResMulti = 0x80000000u;
constexpr uint32_t kResCount = 0x40000000u;

__host__ __device__ constexpr uint32_t res_encode(uint32_t cnt, uint32_t first)
{
    return cnt == 0 ? kResNone
                    : cnt == 1 ? first
                               : (cnt <= 1022u && first < (1u << 20)) ? (kResMulti | kResCount | (cnt << 20) | first)
                                                                      : (kResMulti | first);
}
// The narrow form (2 bytes; at most kRes16MaxP polygons), with the row bitmap
// of pass 1 as pass 1b leaves it (a row's bit stays set iff the point is in
// two or more polygons):
//   bit clear: kRes16None (in no polygon) or q (in exactly polygon q)
//   bit set:   c, the number of polygons (2 <= c <= P); the pairs are written
//              by walking the point's list again
constexpr uint16_t kRes16None = 0xffffu;
constexpr int kHistMax = 11776;             // polygons counted in shared memory (46 KB)


// ------------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t lanemask_lt()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}
// L2 eviction policies: the index stays resident (evict_last) while the
// streamed points pass through (evict_first).
__device__ __forceinline__ uint64_t policy_evict_last()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// The join's passes read the index words of polygons past L1: once per point, at
// random, 32 lines a warp (100M points x 2000 cells 571 -> 549 us, count x 5000 cells
// 497 -> 467, 20M x 1024 queries 703 -> 673).  The others take an L1 line: disk lists
// are read word after word, rows of a clustered table share words, and where points
// crowd into few cells their words are in L1 (past it, 20M points, 90 % of them in 256
// cells of 64 disks, joined in 586 us instead of 257).
template <bool L1 = true>
__device__ __forceinline__ uint32_t ld_idx(const uint32_t *p, uint64_t pol)
{
    uint32_t v;
    if (L1)
        asm volatile("ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
    else
        asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.u32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(pol));
    return v;
}
// The same where `on`, else v stays; without a branch.
template <bool L1>
__device__ __forceinline__ void ld_idx_if(uint32_t &v, const uint32_t *p, uint64_t pol, bool on)
{
    if (L1)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t"
                     "@p ld.global.nc.L2::cache_hint.u32 %0, [%1], %2;\n\t}"
                     : "+r"(v)
                     : "l"(p), "l"(pol), "r"((uint32_t)on));
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t"
                     "@p ld.global.nc.L1::no_allocate.L2::cache_hint.u32 %0, [%1], %2;\n\t}"
                     : "+r"(v)
                     : "l"(p), "l"(pol), "r"((uint32_t)on));
}
__device__ __forceinline__ uint4 ld_idx(const uint4 *p, uint64_t pol)
{
    uint4 v;
    asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ int4 ld_idx(const int4 *p, uint64_t pol)
{
    int4 v;
    asm volatile("ld.global.nc.L2::cache_hint.v4.s32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p), "l"(pol));
    return v;
}
// Bulk prefetch of `bytes` (a multiple of 16) at p (16-byte aligned) into L2
// by the TMA engine: one instruction, no registers, nothing to wait for.
__device__ __forceinline__ void prefetch_l2_bulk(const void *p, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
// mbarrier and 1-D TMA bulk copy (global -> shared) for a warp's own staging
// buffer.  The barrier counts one arrival (the expect_tx of the issuing lane)
// plus the bytes the copy delivers.
__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// dst, src 16-byte aligned; bytes a multiple of 16.  The generic-proxy reads
// of dst that came before are ordered before the copy's writes.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// Waits for the phase of `bar` with the given parity to complete, at most
// max_tries polls (each may suspend the thread for a short time); false if it
// gave up.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint32_t max_tries)
{
    const uint32_t a = smem_u32(bar);
    for (uint32_t t = 0; t < max_tries; ++t) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(a), "r"(parity)
                     : "memory");
        if (done)
            return true;
    }
    return false;
}
constexpr uint32_t kWaitTries = 1u << 22; // polls of a bounded wait before it reports kErrTimeout
constexpr int kWaveWords = 64; // shared words per warp of walk_list_wave: the parities of two entries per lane
// Prefetch of the line holding p into L2.
__device__ __forceinline__ void prefetch_l2(const void *p)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}
// ------------------------------------------------------------- the predicate
// sign of d = (bx-ax)(py-ay) - (by-ay)(px-ax)
template <bool FP32>
__device__ __forceinline__ int orient_sign(int ax, int ay, int bx, int by, int px, int py, uint32_t &esc)
{
    const int dx1 = bx - ax, dy1 = py - ay, dy2 = by - ay, dx2 = px - ax;
    if (FP32) {
        const float t1 = __fmul_rn(__int2float_rn(dx1), __int2float_rn(dy1));
        const float t2 = __fmul_rn(__int2float_rn(dy2), __int2float_rn(dx2));
        const float df = __fsub_rn(t1, t2);
        const float E = __fmul_rn(__fadd_rn(fabsf(t1), fabsf(t2)), 4.76837158203125e-07f); // 2^-21
        if (fabsf(df) > E)
            return df > 0.f ? 1 : -1;
        ++esc;
    }
    const long long d = (long long)dx1 * dy1 - (long long)dy2 * dx2;
    return (d > 0) - (d < 0);
}

// Parity of the crossings of the rightward ray from (px, py) with a fine-row
// edge list sorted by max x descending.  Edges are loaded RW at a time so a
// list costs one L2 round trip per RW edges.
template <bool FP32>
__device__ __forceinline__ uint32_t row_parity(const int4 *__restrict__ e, uint32_t n, int px, int py,
                                               uint32_t &tests, uint32_t &esc, uint64_t pol)
{
    constexpr int RW = 4;
    uint32_t par = 0;
    for (uint32_t k = 0; k < n; k += RW) {
        int4 v[RW];
#pragma unroll
        for (int j = 0; j < RW; ++j)
            v[j] = (k + j < n) ? ld_idx(e + k + j, pol) : make_int4(INT_MIN, 0, INT_MIN, 0);
        bool stop = false;
#pragma unroll
        for (int j = 0; j < RW; ++j) {
            if (stop || max(v[j].x, v[j].z) <= px) {
                stop = true; // this and every later edge ends left of p: no crossing right of p
                continue;
            }
            if ((v[j].y > py) == (v[j].w > py))
                continue; // does not straddle
            if (min(v[j].x, v[j].z) > px) {
                par ^= 1u; // the crossing lies right of p
                continue;
            }
            ++tests;
            const int s = orient_sign<FP32>(v[j].x, v[j].y, v[j].z, v[j].w, px, py, esc);
            par ^= uint32_t((s != 0) & ((s > 0) == (v[j].w > v[j].y)));
        }
        if (stop)
            break;
    }
    return par;
}

// Bounds checks of the index walks, compiled in by SPX_BOUNDS_CHECK (a debug
// build): an offset or id read from the index that points outside its array
// sets kErrInternal in the error word, and the walk treats the point as in no
// polygon of that list instead of reading there.  The host reports the word
// as SPX_EKERNEL.  In the default build the checks compile to nothing.
__device__ __forceinline__ bool in_bounds(bool ok, const IndexView &ix)
{
#ifdef SPX_BOUNDS_CHECK
    if (!ok)
        atomicOr(ix.err, kErrInternal);
    return ok;
#else
    (void)ok;
    (void)ix;
    return true;
#endif
}

// An entry's edges: in the row lists, or (kLocalEdge) in the local ones.
__device__ __forceinline__ const int4 *edge_at(const IndexView &ix, uint32_t y)
{
    return (y & ix.loc_bit) ? ix.loc + (y & ~kLocalEdge) : ix.edge + y;
}
__device__ __forceinline__ bool edges_ok(const IndexView &ix, const uint4 &en)
{
    return !(en.w & kEntBoundary) ||
           ((en.y & ix.loc_bit) ? (uint64_t)(en.y & ~kLocalEdge) + en.z <= ix.n_loc : (uint64_t)en.y + en.z < ix.n_edge);
}

template <bool L1 = true>
__device__ __forceinline__ uint32_t coarse_word(const IndexView &ix, uint32_t px, uint32_t py, uint64_t pol)
{
    return ld_idx<L1>(ix.cell + (((py >> ix.sc) << ix.gc) | (px >> ix.sc)), pol);
}
template <bool L1 = true>
__device__ __forceinline__ uint32_t fine_word(const IndexView &ix, uint32_t w, uint32_t px, uint32_t py,
                                              uint64_t pol)
{
    const uint32_t fm = (1u << ix.sb) - 1;
    if (!in_bounds(((uint64_t)(w & kPayloadMask) + 1) << (2 * ix.sb) <= ix.n_fine, ix))
        return 0u;
    return ld_idx<L1>(ix.fine + (((w & kPayloadMask) << (2 * ix.sb)) | (((py >> ix.sf) & fm) << ix.sb) |
                             ((px >> ix.sf) & fm)),
                  pol);
}
// What an index's entry lists hold: polygons with crossing edges, buffered
// polygons with edges that may be near, or disks.
constexpr int kPoly = 0, kNear = 1, kDisk = 2;

// Resolved word of an in-box point: kind 0 none, 1 one INSIDE polygon, 2 list (a disk
// index has one level, whose words are that already).
template <int KIND = kPoly, bool L1 = true>
__device__ __forceinline__ uint32_t resolve(const IndexView &ix, uint32_t px, uint32_t py, uint64_t pol)
{
    const uint32_t w = coarse_word<L1>(ix, px, py, pol);
    return KIND != kDisk && (w >> 30) == kCellSub ? fine_word<L1>(ix, w, px, py, pol) : w;
}

// One edge's contribution to the crossing parity of (px, py).
template <bool FP32>
__device__ __forceinline__ uint32_t edge_cross(const int4 &v, int px, int py, uint32_t &tests, uint32_t &esc)
{
    if ((v.y > py) == (v.w > py))
        return 0u; // does not straddle
    if (min(v.x, v.z) > px)
        return 1u; // the crossing lies right of p
    if (max(v.x, v.z) <= px)
        return 0u; // the crossing lies at or left of p
    ++tests;
    const int s = orient_sign<FP32>(v.x, v.y, v.z, v.w, px, py, esc);
    return uint32_t((s != 0) & ((s > 0) == (v.w > v.y)));
}

// Membership of (px, py) in one entry's polygon, given the entry's first four
// edges (already loaded; missing ones never straddle).  Longer lists continue
// in row order.
template <bool FP32>
__device__ __forceinline__ uint32_t entry_in(const IndexView &ix, const uint4 &en, const int4 (&v)[4], int px, int py,
                                             uint32_t &tests, uint32_t &esc, uint64_t pol)
{
    if (!(en.w & kEntBoundary))
        return 1u;
    uint32_t par = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        par ^= edge_cross<FP32>(v[j], px, py, tests, esc);
    if (en.z > 4 && max(v[3].x, v[3].z) > px)
        par ^= row_parity<FP32>(edge_at(ix, en.y) + 4, en.z - 4, px, py, tests, esc, pol);
    return par;
}

// Calls f(polygon) for every polygon of the entry list starting at e that
// contains (px, py), ascending.  Entries are taken two at a time: both
// entries in one round trip, then the first four edges of each in another
// (the entry array ends with sentinels, so reading two is in bounds).
template <bool FP32, class F>
__device__ __forceinline__ void walk_entries(const IndexView &ix, const uint4 *e, int px, int py, uint32_t &tests,
                                             uint32_t &esc, uint64_t pol, F f)
{
    constexpr int B = 2;
    for (bool more = true; more; e += B) {
        if (!in_bounds((uint64_t)(e - ix.ent) + 1 < ix.n_ent, ix))
            return;
        uint4 en[B];
#pragma unroll
        for (int k = 0; k < B; ++k)
            en[k] = ld_idx(e + k, pol);
#pragma unroll
        for (int k = 0; k < B; ++k)
            if ((k == 0 || !(en[0].w & kEntLast)) &&
                !in_bounds(en[k].x < ix.P && edges_ok(ix, en[k]),
                           ix))
                return;
        // entries of this list among the B: up to and including the first LAST
        uint32_t live = 0;
#pragma unroll
        for (int k = 0; k < B; ++k) {
            if (more)
                live |= 1u << k;
            if (more && (en[k].w & kEntLast))
                more = false;
        }
        int4 v[B][4];
#pragma unroll
        for (int k = 0; k < B; ++k) {
            const uint32_t nk = ((live >> k) & 1u) && (en[k].w & kEntBoundary) ? min(en[k].z, 4u) : 0u;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                v[k][j] = ld_idx((uint32_t)j < nk ? edge_at(ix, en[k].y) + j : ix.edge, pol);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if ((uint32_t)j >= nk)
                    v[k][j] = make_int4(0, 0, 0, 0);
        }
#pragma unroll
        for (int k = 0; k < B; ++k)
            if (((live >> k) & 1u) && entry_in<FP32>(ix, en[k], v[k], px, py, tests, esc, pol))
                f(en[k].x);
    }
}

// Calls f(polygon) for every polygon containing the in-box point (px, py),
// ascending (only called for points with more than one match: their word is a list).
template <bool FP32, class F>
__device__ __forceinline__ void point_emit(const IndexView &ix, int px, int py, uint64_t pol, F f)
{
    uint32_t t = 0, s = 0;
    const uint32_t w = resolve(ix, (uint32_t)px, (uint32_t)py, pol);
    if ((w >> 30) != kCellList)
        return;
    walk_entries<FP32>(ix, ix.ent + (w & kPayloadMask), px, py, t, s, pol, f);
}

// Walk an entry list: number of polygons containing (px, py), smallest id.
// Written so that the lanes of a warp stay converged around every load: the
// common case (at most two entries, at most four edges each) issues all its
// loads unconditionally, from clamped addresses that always lie inside the
// arrays (both end with a sentinel), and selects the results; divergent lanes
// of a warp would otherwise serialise their memory round trips.  Longer lists
// finish in a loop.
template <bool FP32>
__device__ __forceinline__ uint32_t walk_list(const IndexView &ix, uint32_t e0, int px, int py, uint32_t &first,
                                              uint32_t &tests, uint32_t &esc, uint64_t pol)
{
    if (!in_bounds((uint64_t)e0 + 1 < ix.n_ent, ix))
        return 0u;
    const uint4 *e = ix.ent + e0;
    const uint4 en0 = ld_idx(e, pol), en1 = ld_idx(e + 1, pol);
    const bool two = !(en0.w & kEntLast);
    if (!in_bounds(en0.x < ix.P && edges_ok(ix, en0) &&
                       (!two || (en1.x < ix.P && edges_ok(ix, en1))),
                   ix))
        return 0u;
    const uint32_t n0 = (en0.w & kEntBoundary) ? min(en0.z, 4u) : 0u;
    const uint32_t n1 = (two && (en1.w & kEntBoundary)) ? min(en1.z, 4u) : 0u;
    int4 v0[4], v1[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        v0[j] = ld_idx((uint32_t)j < n0 ? edge_at(ix, en0.y) + j : ix.edge, pol);
        v1[j] = ld_idx((uint32_t)j < n1 ? edge_at(ix, en1.y) + j : ix.edge, pol);
    }
    uint32_t p0 = 0, p1 = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t c0 = edge_cross<FP32>(v0[j], px, py, tests, esc);
        const uint32_t c1 = edge_cross<FP32>(v1[j], px, py, tests, esc);
        p0 ^= (uint32_t)j < n0 ? c0 : 0u;
        p1 ^= (uint32_t)j < n1 ? c1 : 0u;
    }
    // lists longer than four edges: the rest, in row order
    if ((en0.w & kEntBoundary) && en0.z > 4 && max(v0[3].x, v0[3].z) > px)
        p0 ^= row_parity<FP32>(edge_at(ix, en0.y) + 4, en0.z - 4, px, py, tests, esc, pol);
    if (two && (en1.w & kEntBoundary) && en1.z > 4 && max(v1[3].x, v1[3].z) > px)
        p1 ^= row_parity<FP32>(edge_at(ix, en1.y) + 4, en1.z - 4, px, py, tests, esc, pol);
    const uint32_t in0 = (en0.w & kEntBoundary) ? p0 : 1u;
    const uint32_t in1 = two ? ((en1.w & kEntBoundary) ? p1 : 1u) : 0u;
    uint32_t c = in0 + in1;
    first = in0 ? en0.x : en1.x;
    if (two && !(en1.w & kEntLast)) {
        // three or more polygons share this fine cell (rare)
        for (const uint4 *q = e + 2;; ++q) {
            if (!in_bounds((uint64_t)(q - ix.ent) < ix.n_ent, ix))
                break;
            const uint4 en = ld_idx(q, pol);
            if (!in_bounds(en.x < ix.P && edges_ok(ix, en), ix))
                break;
            if (!(en.w & kEntBoundary) || row_parity<FP32>(edge_at(ix, en.y), en.z, px, py, tests, esc, pol)) {
                if (!c)
                    first = en.x;
                ++c;
            }
            if (en.w & kEntLast)
                break;
        }
    }
    return c;
}

// A point is within distance r of a centre c iff (px-cx)^2 + (py-cy)^2 <= r^2,
// exact in int64 (differences < 2^31; r < 2^30; the x term is compared with
// r^2 before the sum, so the sum cannot overflow).
__device__ __forceinline__ bool in_disk(const int4 &d, int px, int py)
{
    const long long dx = (long long)px - d.x, dy = (long long)py - d.y, rr = (long long)d.z * d.z;
    const long long dx2 = dx * dx;
    return dx2 <= rr && dx2 + dy * dy <= rr;
}

// Does polygon q of its own index hold the in-box point (px, py)?
template <bool FP32>
__device__ __noinline__ bool poly_holds(const IndexView &ix, uint32_t q, int px, int py, uint32_t &tests, uint32_t &esc,
                                        uint64_t pol)
{
    const uint32_t w = resolve(ix, (uint32_t)px, (uint32_t)py, pol), pay = w & kPayloadMask;
    if ((w >> 30) == kCellInsideOne)
        return pay == q;
    if ((w >> 30) != kCellList)
        return false;
    for (uint64_t e = pay; in_bounds(e < ix.n_ent, ix); ++e) {
        const uint4 en = ld_idx(ix.ent + e, pol);
        if (en.x == q && in_bounds(edges_ok(ix, en), ix))
            return !(en.w & kEntBoundary) || row_parity<FP32>(edge_at(ix, en.y), en.z, px, py, tests, esc, pol);
        if (en.x >= q || (en.w & kEntLast))
            return false;
    }
    return false;
}

// The polygons of an entry list that contain a point, for the 32 lanes of a
// converged warp at once, each lane with its own point (px, py) and list
// (starting at entry e0; has = false: the lane takes part but has none).
// Calls f(q) on each lane, in ascending q, for every polygon q of its list
// that contains its point.  The entries are taken two per lane per wave (one
// round trip); the edges of all the wave's boundary entries of all lanes are
// then tested by the whole warp, 64 at a time: edge k of the flattened list
// goes to lane k mod 32, which finds the lane that owns it by a binary search
// over the lanes' prefix sums, tests that lane's point, and XORs the crossing
// into that lane's parity in shared memory.  Lanes never loop on their own
// long lists (which would diverge and run one dependent load per step); the
// sorted lists' early stop is not used (an edge that ends left of the point
// counts nothing; recording where each list could stop measured slower).
// s_par: kWaveWords words of shared memory owned by this warp.
// KIND kNear: the list is one of a buffered index (nv).  An edge hits when it comes
// within its polygon's radius of the point, hits are ORed instead of XORed, and
// a point that no edge hits asks the polygons' own index where the entry says
// that the boundary may cross the cell.
template <bool FP32, int KIND = kPoly, class F>
__device__ __forceinline__ void walk_list_wave(const IndexView &ix, bool has, uint32_t e0, int px, int py,
                                               uint32_t &tests, uint32_t &esc, uint64_t pol, uint32_t *s_par, F f,
                                               const NearView *nv = nullptr)
{
    if constexpr (KIND == kDisk) { // short lists of disks, a test each: every lane walks its own
        const uint32_t n = has ? ld_idx(nv->dent + e0, pol) : 0u;
        for (uint32_t k = 1; k <= n; ++k) {
            const uint32_t en = ld_idx(nv->dent + e0 + k, pol), q = en >> 1;
            tests += en & 1u;
            if (!(en & 1u) || in_disk(__ldg(nv->disk + q), px, py))
                f(q);
        }
        __syncwarp();
        return;
    }
    const int lane = threadIdx.x & 31;
    const uint4 *e = ix.ent + (has ? e0 : 0u);
    bool more = has;
    while (__any_sync(kFull, more)) {
        more = more && in_bounds((uint64_t)(e - ix.ent) + 1 < ix.n_ent, ix);
        // two entries (the entry array ends with sentinels: reading e + 1 is in bounds)
        uint4 ea = more ? ld_idx(e, pol) : make_uint4(0, 0, 0, kEntLast);
        const uint4 eb0 = more ? ld_idx(e + 1, pol) : make_uint4(0, 0, 0, kEntLast);
        const bool hb0 = more && !(ea.w & kEntLast);
        if (more && !in_bounds(ea.x < ix.P && edges_ok(ix, ea) &&
                                   (!hb0 || (eb0.x < ix.P &&
                                             edges_ok(ix, eb0))),
                               ix)) {
            more = false; // this lane's list ends here
            ea = make_uint4(0, 0, 0, kEntLast);
        }
        const bool hb = more && !(ea.w & kEntLast);
        const uint4 eb = hb ? eb0 : make_uint4(0, 0, 0, kEntLast);
        const uint32_t za = (more && (ea.w & kEntBoundary)) ? ea.z : 0u;
        const uint32_t zb = (hb && (eb.w & kEntBoundary)) ? eb.z : 0u;
        const uint32_t tot = za + zb;
        int ra = 0, rb = 0; // kNear: the entries' radii
        if (KIND == kNear) {
            ra = za ? __ldg(nv->rad + ea.x) : 0;
            rb = zb ? __ldg(nv->rad + eb.x) : 0;
        }
        uint32_t pa = 0, pb = 0;
        if (__any_sync(kFull, tot != 0)) {
            uint32_t incl = tot;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, incl, o);
                if (lane >= o)
                    incl += t;
            }
            const uint32_t T = __shfl_sync(kFull, incl, 31);
            s_par[lane] = 0u;
            s_par[32 + lane] = 0u;
            __syncwarp();
            for (uint32_t base = 0; base < T; base += 64) {
                int4 v[2];
                uint32_t slot[2], own[2];
                int ox[2], oy[2], rad[2];
                bool act[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const uint32_t k = base + 32 * h + lane;
                    act[h] = k < T;
                    uint32_t o = 0; // the owner: the first lane whose inclusive prefix exceeds k
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1)
                        if (__shfl_sync(kFull, incl, o + step - 1) <= k)
                            o += step;
                    o = act[h] ? o : 0u;
                    const uint32_t oi = __shfl_sync(kFull, incl, o), ot = __shfl_sync(kFull, tot, o);
                    const uint32_t oza = __shfl_sync(kFull, za, o);
                    const uint32_t oya = __shfl_sync(kFull, ea.y, o), oyb = __shfl_sync(kFull, eb.y, o);
                    ox[h] = __shfl_sync(kFull, px, o);
                    oy[h] = __shfl_sync(kFull, py, o);
                    const uint32_t t = k - (oi - ot);
                    slot[h] = t >= oza ? 1u : 0u;
                    own[h] = o;
                    if (KIND == kNear) {
                        const int r0 = __shfl_sync(kFull, ra, o), r1 = __shfl_sync(kFull, rb, o);
                        rad[h] = slot[h] ? r1 : r0;
                    }
                    const uint32_t ei = slot[h] ? oyb + (t - oza) : oya + t;
                    v[h] = act[h] ? ld_idx(edge_at(ix, ei), pol) : make_int4(0, 0, 0, 0); // a zero edge never straddles
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (KIND == kNear) {
                        if (act[h] && seg_near<FP32>(v[h], ox[h], oy[h], rad[h]))
                            atomicOr(s_par + 32 * slot[h] + own[h], 1u);
                    } else if (act[h] && edge_cross<FP32>(v[h], ox[h], oy[h], tests, esc)) {
                        atomicXor(s_par + 32 * slot[h] + own[h], 1u);
                    }
                }
            }
            __syncwarp();
            pa = s_par[lane];
            pb = s_par[32 + lane];
            __syncwarp(); // s_par is rewritten by the next wave
        }
        if (KIND == kNear) {
            if (more && !pa && (ea.w & kEntCross))
                pa = poly_holds<FP32>(nv->in, ea.x, px, py, tests, esc, pol);
            if (hb && !pb && (eb.w & kEntCross))
                pb = poly_holds<FP32>(nv->in, eb.x, px, py, tests, esc, pol);
        }
        if (more && (!(ea.w & kEntBoundary) || pa))
            f(ea.x);
        if (hb && (!(eb.w & kEntBoundary) || pb))
            f(eb.x);
        more = hb && !(eb.w & kEntLast);
        e += 2;
    }
}

// Shared-memory histogram update for one item of every lane of a converged
// warp (lanes with has = false add nothing).  Clustered points often put the
// whole warp on one polygon: then one atomic adds the lane count.
__device__ __forceinline__ void hist_add_warp(uint32_t *h, bool has, uint32_t q)
{
    const uint32_t m = __ballot_sync(kFull, has);
    if (!m)
        return;
    const uint32_t qmin = __reduce_min_sync(kFull, has ? q : 0xffffffffu);
    const uint32_t qmax = __reduce_max_sync(kFull, has ? q : 0u);
    if (qmin == qmax) {
        if ((int)(threadIdx.x & 31) == __ffs(m) - 1)
            atomicAdd(h + qmin, (uint32_t)__popc(m));
    } else if (has) {
        atomicAdd(h + q, 1u);
    }
}

// Global counter update for one item of every lane of a converged warp (lanes
// with has = false add nothing): one atomic per distinct polygon of the warp,
// so a clustered table's lanes do not serialise on the same counter.
__device__ __forceinline__ void global_add_warp(unsigned long long *cnt, bool has, uint32_t q)
{
    const uint32_t m = __ballot_sync(kFull, has);
    if (!m)
        return;
    // all lanes on one polygon (clustered tables): one atomic, no match
    const uint32_t qmin = __reduce_min_sync(kFull, has ? q : 0xffffffffu);
    const uint32_t qmax = __reduce_max_sync(kFull, has ? q : 0u);
    if (qmin == qmax) {
        if ((int)(threadIdx.x & 31) == __ffs(m) - 1)
            atomicAdd(cnt + qmin, (unsigned long long)__popc(m));
        return;
    }
    const uint32_t peers = __match_any_sync(kFull, has ? q : 0xffffffffu);
    if (has && (int)(threadIdx.x & 31) == __ffs(peers) - 1)
        atomicAdd(cnt + q, (unsigned long long)__popc(peers));
}

// Whole predicate for one point (plain kernels, overflow path).
template <bool FP32>
__device__ __forceinline__ uint32_t point_count(const IndexView &ix, int px, int py, uint32_t &first,
                                                uint32_t &tests, uint32_t &esc, uint64_t pol)
{
    if ((unsigned)px >= kBox || (unsigned)py >= kBox)
        return 0;
    const uint32_t w = resolve(ix, (uint32_t)px, (uint32_t)py, pol);
    const uint32_t kind = w >> 30;
    if (kind == kCellEmpty)
        return 0;
    if (kind == kCellInsideOne) {
        first = w & kPayloadMask;
        return 1;
    }
    return walk_list<FP32>(ix, w & kPayloadMask, px, py, first, tests, esc, pol);
}

// The number of buffered polygons that the in-box point (px, py) meets, by one
// lane (points whose count does not fit their 32-bit result).
template <bool FP32>
__device__ __noinline__ uint32_t near_count(const IndexView &ix, const NearView &nv, int px, int py, uint64_t pol)
{
    const uint32_t w = resolve(ix, (uint32_t)px, (uint32_t)py, pol);
    uint32_t n = 0, t = 0, s = 0;
    if ((w >> 30) < kCellList)
        return (w >> 30) == kCellInsideOne ? 1u : 0u;
    for (uint64_t e = w & kPayloadMask; in_bounds(e < ix.n_ent, ix); ++e) {
        const uint4 en = ld_idx(ix.ent + e, pol);
        bool hit = !(en.w & kEntBoundary);
        if (in_bounds(en.x < ix.P && (hit || (uint64_t)en.y + en.z < ix.n_edge), ix))
            for (uint32_t k = 0; k < en.z && !hit; ++k)
                hit = seg_near<FP32>(ld_idx(ix.edge + en.y + k, pol), px, py, __ldg(nv.rad + en.x));
        n += hit || ((en.w & kEntCross) && poly_holds<FP32>(nv.in, en.x, px, py, t, s, pol)) ? 1u : 0u;
        if (en.w & kEntLast)
            break;
    }
    return n;
}

// The number of disks that hold the in-box point (px, py), by one lane.
__device__ __noinline__ uint32_t disk_count(const IndexView &ix, const NearView &nv, int px, int py, uint64_t pol)
{
    const uint32_t w = coarse_word(ix, (uint32_t)px, (uint32_t)py, pol);
    if ((w >> 30) < kCellList)
        return (w >> 30) == kCellInsideOne ? 1u : 0u;
    const uint32_t *e = nv.dent + (w & kPayloadMask);
    uint32_t c = 0;
    for (uint32_t n = ld_idx(e, pol), k = 1; k <= n; ++k) {
        const uint32_t en = ld_idx(e + k, pol);
        c += !(en & 1u) || in_disk(__ldg(nv.disk + (en >> 1)), px, py) ? 1u : 0u;
    }
    return c;
}

__device__ __forceinline__ unsigned long long warp_sum64(unsigned long long v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Adds a CTA's counters to the ctx's, once per CTA (every thread of the CTA calls
// it, at the end): with an atomic per warp and counter a persistent kernel ended in
// 15,000 atomics on two cache lines.
__device__ __forceinline__ void add_stats(unsigned long long *stats, uint32_t pts, uint32_t tests, uint32_t esc,
                                          uint32_t pairs)
{
    __shared__ unsigned long long s_stat[4];
    if (threadIdx.x < 4)
        s_stat[threadIdx.x] = 0ull;
    __syncthreads();
    const unsigned long long v[4] = {warp_sum64(pts), warp_sum64(tests), warp_sum64(esc), warp_sum64(pairs)};
    if ((threadIdx.x & 31) == 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (v[k])
                atomicAdd(s_stat + k, v[k]);
    }
    __syncthreads();
    static_assert(kStatPoints == 0 && kStatTests == 1 && kStatEscalations == 2 && kStatPairs == 3, "order of the counters");
    if (threadIdx.x < 4 && s_stat[threadIdx.x])
        atomicAdd(stats + threadIdx.x, s_stat[threadIdx.x]);
}

template <class K>
int persistent_grid(K kernel, int threads, size_t smem, uint32_t ntiles)
{
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
    if (per_sm < 1)
        per_sm = 1;
    int grid = per_sm * device_sm_count();
    if ((uint32_t)grid > ntiles)
        grid = (int)ntiles;
    return grid;
}

// ------------------------------------------------------- plain comparison join
// Exact int64 only; one thread per point; pass 1 counts per 256-point block,
// a one-block scan makes block offsets, pass 2 recounts and writes.  Counts by
// global atomics.
__global__ void __launch_bounds__(kPlainThreads) k_plain_count(JoinLaunch a, unsigned long long *block_cnt)
{
    __shared__ uint32_t s_w[(kPlainThreads / 32)];
    const uint64_t idx = (uint64_t)blockIdx.x * kPlainThreads + threadIdx.x;
    uint32_t c = 0, first = 0, t = 0, e = 0;
    if (idx < a.n) {
        const int2 p = a.pts[idx];
        c = point_count<false>(a.ix, p.x, p.y, first, t, e, policy_evict_last());
    }
    uint32_t s = c;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        s += __shfl_xor_sync(kFull, s, o);
    if ((threadIdx.x & 31) == 0)
        s_w[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long b = 0;
        for (int w = 0; w < (kPlainThreads / 32); ++w)
            b += s_w[w];
        block_cnt[blockIdx.x] = b;
    }
}

// Exclusive scan by blocks of 1024 threads, kScanChunk values per step.  A warp
// takes 256 consecutive values as eight rows of 32, so its loads and stores are
// whole lines (eight consecutive values per thread touched 16 lines per access:
// 67M values 399 -> 163 us in k_scan_apply, 11,719 values 14.4 -> 7.7 us in
// k_scan, where one SM's L1 does it all).
constexpr int kScanItems = 8;
constexpr uint64_t kScanChunk = 1024 * kScanItems;

// Loads this thread's values of the step that starts at v[b]: row j of warp w
// is v[b + 256 w + 32 j ..].
__device__ __forceinline__ void scan_load(const unsigned long long *v, uint64_t b, uint64_t n,
                                          unsigned long long (&x)[kScanItems])
{
    const uint64_t i0 = b + (threadIdx.x >> 5) * (32 * kScanItems) + (threadIdx.x & 31);
#pragma unroll
    for (int j = 0; j < kScanItems; ++j)
        x[j] = i0 + 32 * j < n ? v[i0 + 32 * j] : 0ull;
}

// Turns the values of a step into their exclusive prefixes within the step
// (x[j] becomes the prefix) and returns the step's sum.  s_w: 33 words.
__device__ __forceinline__ unsigned long long scan_step(unsigned long long (&x)[kScanItems], unsigned long long *s_w)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long any = 0, wsum = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j)
        any |= x[j];
    if (!__any_sync(kFull, (any >> 27) != 0)) { // a row's sum fits 32 bits
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) {
            const uint32_t v = (uint32_t)x[j];
            uint32_t inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(kFull, inc, o);
                if (lane >= o)
                    inc += t;
            }
            x[j] = wsum + (inc - v);
            wsum += __shfl_sync(kFull, inc, 31);
        }
    } else {
#pragma unroll 1
        for (int j = 0; j < kScanItems; ++j) {
            unsigned long long v = 0, inc;
#pragma unroll
            for (int k = 0; k < kScanItems; ++k) // x stays in registers
                v = k == j ? x[k] : v;
            inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long t = __shfl_up_sync(kFull, inc, o);
                if (lane >= o)
                    inc += t;
            }
#pragma unroll
            for (int k = 0; k < kScanItems; ++k)
                x[k] = k == j ? wsum + (inc - v) : x[k];
            wsum += __shfl_sync(kFull, inc, 31);
        }
    }
    if (lane == 0)
        s_w[warp] = wsum;
    __syncthreads();
    if (warp == 0) {
        const unsigned long long w = s_w[lane];
        unsigned long long wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long t = __shfl_up_sync(kFull, wi, o);
            if (lane >= o)
                wi += t;
        }
        s_w[lane] = wi - w;
        if (lane == 31)
            s_w[32] = wi;
    }
    __syncthreads();
    const unsigned long long before = s_w[warp], total = s_w[32];
#pragma unroll
    for (int j = 0; j < kScanItems; ++j)
        x[j] += before;
    __syncthreads(); // s_w is rewritten by the next step
    return total;
}

__device__ __forceinline__ void scan_store(unsigned long long *v, uint64_t b, uint64_t n, unsigned long long base,
                                           const unsigned long long (&x)[kScanItems])
{
    const uint64_t i0 = b + (threadIdx.x >> 5) * (32 * kScanItems) + (threadIdx.x & 31);
#pragma unroll
    for (int j = 0; j < kScanItems; ++j)
        if (i0 + 32 * j < n)
            v[i0 + 32 * j] = base + x[j];
}

// One block, the steps one after the other with a carried total.
__global__ void __launch_bounds__(1024) k_scan(unsigned long long *v, uint64_t n, unsigned long long *total)
{
    __shared__ unsigned long long s_w[33];
    unsigned long long carry = 0, x[kScanItems];
    for (uint64_t b = 0; b < n; b += kScanChunk) {
        scan_load(v, b, n, x);
        const unsigned long long t = scan_step(x, s_w);
        scan_store(v, b, n, carry, x);
        carry += t;
    }
    if (threadIdx.x == 0 && total)
        *total = carry;
}

// Device-wide exclusive scan for long arrays: per-chunk sums, a one-block scan
// of the sums, then every chunk rescanned from its base.
__global__ void __launch_bounds__(1024) k_scan_partials(const unsigned long long *v, uint64_t n,
                                                        unsigned long long *part)
{
    __shared__ unsigned long long s_w[32];
    unsigned long long x[kScanItems], sum = 0;
    scan_load(v, (uint64_t)blockIdx.x * kScanChunk, n, x);
#pragma unroll
    for (int j = 0; j < kScanItems; ++j)
        sum += x[j];
    sum = warp_sum64(sum);
    if ((threadIdx.x & 31) == 0)
        s_w[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x < 32) {
        sum = warp_sum64(s_w[threadIdx.x]);
        if (threadIdx.x == 0)
            part[blockIdx.x] = sum;
    }
}

__global__ void __launch_bounds__(1024) k_scan_apply(unsigned long long *v, uint64_t n,
                                                     const unsigned long long *part_off)
{
    __shared__ unsigned long long s_w[33];
    const uint64_t b = (uint64_t)blockIdx.x * kScanChunk;
    unsigned long long x[kScanItems];
    scan_load(v, b, n, x);
    scan_step(x, s_w);
    scan_store(v, b, n, part_off[blockIdx.x], x);
}

__device__ __forceinline__ uint32_t warp_sum32(uint32_t v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// ---------------------------------------------- count-only aggregate
// The count-only aggregation that never materialises the join (§5.2 "Spatial
// Aggregations").  No CTA barrier in its loop: every warp works alone on
// chunks of 32 x kWItems consecutive points (chunk c goes to warp c mod
// #warps), loads its points with coalesced 8-byte loads, resolves the coarse
// and fine words of all of a lane's points with independent loads, and queues
// its list points in a per-warp shared-memory queue that it walks 32 at a time
// once the whole chunk is resolved (the chunk's points and words are dead by
// then, which keeps the kernel at 64 registers and 4 CTAs per SM).  A warp
// never waits for another warp, so a slow walk or an index miss only stalls
// its own warp.  The chunks (256 points) are those of the join's passes.
#ifndef SPX_WARP_ITEMS
#define SPX_WARP_ITEMS 8
#endif
#ifndef SPX_WARP_MIN_BLOCKS
#define SPX_WARP_MIN_BLOCKS 4
#endif
constexpr int kWItems = SPX_WARP_ITEMS; // points per lane per chunk (8: 256-point chunks)
constexpr int kWChunk = 32 * kWItems;   // consecutive points per warp chunk
constexpr int kWQueue = kWChunk;        // list points queued per warp: a whole chunk
// per warp: the queue, then the words of walk_list_wave
constexpr size_t kWarpSmem = size_t(kWarps) * (kWQueue * sizeof(uint4) + kWaveWords * sizeof(uint32_t));

template <bool FP32, bool CLUSTERED>
__global__ void __launch_bounds__(kThreads, SPX_WARP_MIN_BLOCKS)
    k_warp(JoinLaunch a, uint32_t nchunks, int use_hist)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint4 *s_q = reinterpret_cast<uint4 *>(s_raw) + warp * kWQueue; // (x, y, first entry, chunk index)
    uint32_t *s_par = reinterpret_cast<uint32_t *>(s_raw + size_t(kWarps) * kWQueue * sizeof(uint4)) + warp * kWaveWords;
    uint32_t *s_hist = reinterpret_cast<uint32_t *>(s_raw + kWarpSmem);
    const IndexView &ix = a.ix;
    const uint64_t keep = policy_evict_last();
    const bool hist = use_hist && a.counts;
    if (hist)
        for (uint32_t i = threadIdx.x; i < ix.P; i += kThreads)
            s_hist[i] = 0;
    __syncthreads();
    uint32_t n_tests = 0, n_esc = 0, n_pts = 0, n_pairs = 0;
    // count one polygon for every lane with has (converged warp)
    auto count1 = [&](bool has, uint32_t q) {
        if (!a.counts)
            return;
        if (!hist)
            global_add_warp(a.counts, has, q);
        else if (CLUSTERED) // lanes mostly share a counter: one atomic per distinct polygon
            hist_add_warp(s_hist, has, q);
        else if (has) // lanes mostly hit different counters: one atomic each, no vote
            atomicAdd(s_hist + q, 1u);
    };
    const uint32_t nw = gridDim.x * kWarps;
    for (uint32_t ch = blockIdx.x * kWarps + warp; ch < nchunks; ch += nw) {
        const uint64_t base = (uint64_t)ch * kWChunk;
        const uint32_t npts = (uint32_t)min((uint64_t)kWChunk, a.n - base);
        int2 p[kWItems];
        uint32_t w[kWItems];
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const uint32_t loc = j * 32 + lane;
            p[j] = loc < npts ? __ldcs(a.pts + base + loc) : make_int2(-1, -1);
            n_pts += loc < npts ? 1u : 0u;
        }
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const bool ok = (unsigned)p[j].x < kBox && (unsigned)p[j].y < kBox;
            const uint32_t cw = coarse_word(ix, ok ? (uint32_t)p[j].x : 0u, ok ? (uint32_t)p[j].y : 0u, keep);
            w[j] = ok ? cw : 0u;
        }
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const bool sub = (w[j] >> 30) == kCellSub;
            if (sub)
                w[j] = fine_word(ix, w[j], (uint32_t)p[j].x, (uint32_t)p[j].y, keep);
        }
        uint32_t total = 0, qn = 0;
        // walk m <= 32 queued points starting at k0, one per lane
        auto walk = [&](uint32_t k0, uint32_t m) {
            __syncwarp();
            const bool has = (uint32_t)lane < m;
            const uint4 it = s_q[k0 + (has ? lane : 0)]; // idle lanes walk nothing
            // the warp walks its lanes' lists together; a point's first polygon is
            // counted with the warp below, any further ones at once
            uint32_t f = 0, c = 0;
            walk_list_wave<FP32>(ix, has, it.z, (int)it.x, (int)it.y, n_tests, n_esc, keep, s_par, [&](uint32_t q) {
                if (c == 0)
                    f = q;
                else if (a.counts)
                    hist ? (void)atomicAdd(s_hist + q, 1u) : (void)atomicAdd(a.counts + q, 1ull);
                ++c;
            });
            total += c;
            count1(c >= 1, f);
            __syncwarp();
        };
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const uint32_t kind = w[j] >> 30, loc = j * 32 + lane;
            const bool one = kind == kCellInsideOne && in_bounds((w[j] & kPayloadMask) < ix.P, ix),
                       lst = kind == kCellList;
            total += one ? 1u : 0u;
            count1(one, w[j] & kPayloadMask);
            const uint32_t bl = __ballot_sync(kFull, lst);
            if (lst)
                s_q[qn + __popc(bl & lanemask_lt())] =
                    make_uint4((uint32_t)p[j].x, (uint32_t)p[j].y, w[j] & kPayloadMask, loc);
            qn += __popc(bl);
        }
        for (uint32_t k0 = 0; k0 < qn; k0 += 32)
            walk(k0, min(qn - k0, 32u));
        n_pairs += total;
    }
    if (hist) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < ix.P; i += kThreads)
            if (s_hist[i])
                atomicAdd(a.counts + i, (unsigned long long)s_hist[i]);
    }
    add_stats(a.stats, n_pts, n_tests, n_esc, n_pairs);
}

// ---------------------------------------------- join pass 1 as two kernels
// Pass 1a (k_resolve) is the streaming half of the first pass of the Map:
// every warp takes its own 256-point chunks (chunk c goes to warp c mod
// #warps), loads the points with coalesced 8-byte loads, reads the coarse
// word of every point and, in mixed coarse cells, the fine word, all with
// independent loads, and stores each point's result at once: none, its one
// INSIDE polygon (counted here: §4.3, interior pixels need no test), or, for
// a point whose fine cell holds an entry list, the list's first entry.  Those
// points need the exact boundary test.  Pass 1a marks them in a bitmap over
// the rows: the ballot of the list points of a round of 32 rows is the
// bitmap word of those rows.  It stores each chunk's pair total without
// them.  With no walk in it, the kernel is a short stream of independent
// loads and stores that keeps many warps per SM busy.
//
// Pass 1b (k_walk) runs the exact tests of the marked rows (§4.3 boundary
// index): every warp takes a contiguous range of bitmap words, a lane per
// word, gathers the marked rows into its shared-memory queue and walks them
// in full rounds of 32, one row per lane (the point and its stored first
// entry, two independent loads, then the entry list).  It rewrites the row's
// result, adds the row's pairs to its chunk's total and counts them.
#ifndef SPX_RESOLVE_MIN_BLOCKS
#define SPX_RESOLVE_MIN_BLOCKS 8
#endif
constexpr int kResolveMinBlocks = SPX_RESOLVE_MIN_BLOCKS;
#ifndef SPX_WALK_MIN_BLOCKS
#define SPX_WALK_MIN_BLOCKS 4
#endif
constexpr int kWalkMinBlocks = SPX_WALK_MIN_BLOCKS;
#ifndef SPX_WALK_BATCH
#define SPX_WALK_BATCH 4
#endif
constexpr uint32_t kWalkGroups = 16;
constexpr int kWalkBatch = SPX_WALK_BATCH; // rounds of rows resolved at a time
constexpr int kWalkQueue = 32 * (kWalkBatch + 1); // < 32 carried over + a batch; or a batch less one + a gather step
// With the block summary (SUM), a CTA of 1024 threads (one per SM) first
// copies the summary into shared memory; a point whose block is empty or
// INSIDE one polygon is resolved there and reads no index word.  Random
// 4-byte index loads are what bounds this pass (every lane's word lies in
// another cache line, and the L1 looks up one line at a time), and a
// shared-memory lookup costs a fraction of one.
constexpr int kResolveSumThreads = 1024;
#ifndef SPX_PREFETCH_CHUNKS
#define SPX_PREFETCH_CHUNKS 1
#endif
constexpr int kPrefetchChunks = SPX_PREFETCH_CHUNKS; // L2 prefetch distance of pass 1a, in a warp's chunks
#ifndef SPX_TMA_POINTS
#define SPX_TMA_POINTS 1
#endif
constexpr bool kTmaPoints = SPX_TMA_POINTS != 0; // pass 1a stages points with bulk copies when they fit

// Shared memory of pass 1a: [summary][TMA: per warp a chunk buffer, then per
// warp an mbarrier][counters].
__host__ __device__ constexpr size_t resolve_smem_head(int warps, bool sum, int sg, bool tma)
{
    return (sum ? ((size_t(2) << (2 * sg)) + 15) & ~size_t(15) : 0) +
           (tma ? size_t(warps) * (kWChunk * sizeof(int2) + sizeof(uint64_t)) : 0);
}

// With the summary the kernel is bound by issue (0.65 to 0.74 of the issue slots,
// ALU first), so it is written for few instructions: whole chunks run without
// row checks, a point outside the box reads a masked summary word instead of a
// selected one, loads are predicated instead of branched around, the kind of a
// word is a signed comparison (kind 1: at least 2^30; lists: negative), a counter's
// address is the word shifted left (its kind bits fall off), and lane 0 stores the
// eight ballots.  100M points x 2000 cells: 322 -> 285 us, x 1024 disks 258 -> 213.
// Each warp loads its next chunk's points before the current chunk's words, and
// prefetches the one after into L2.
// OUT says what is kept per point: kOut32 or kOut16 (a result of that width and
// the chunk's pair total), or kOutCount (nothing but the bitmap: the count
// aggregate, whose pass 1b only counts).
constexpr int kOut32 = 0, kOut16 = 1, kOutCount = 2;

template <int OUT, bool DISK>
__global__ void __launch_bounds__(kResolveSumThreads, 1)
    k_resolve_sum(const __grid_constant__ JoinLaunch a, uint32_t *pend, uint32_t nchunks, int use_hist)
{
    constexpr int WARPS = kResolveSumThreads / 32;
    extern __shared__ __align__(16) unsigned char s_raw[];
    const IndexView &ix = a.ix;
    const uint32_t sum_words = 1u << (2 * ix.sg), smask = sum_words - 1u; // 16-bit words
    const uint16_t *s_sum = reinterpret_cast<const uint16_t *>(s_raw);
    uint32_t *s_hist = reinterpret_cast<uint32_t *>(s_raw + resolve_smem_head(WARPS, true, ix.sg, false));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t keep = policy_evict_last();
    const bool hist = use_hist && a.counts;
    const uint32_t nw = gridDim.x * WARPS, hist_at = smem_u32(s_hist);
    for (uint32_t i = threadIdx.x; i < (sum_words + 7) / 8; i += kResolveSumThreads)
        reinterpret_cast<uint4 *>(s_raw)[i] = ld_idx(ix.sum + i, keep);
    if (hist)
        for (uint32_t i = threadIdx.x; i < ix.P; i += kResolveSumThreads)
            s_hist[i] = 0;
    __syncthreads();
    uint32_t n_pairs = 0;
    int2 pn[kWItems]; // the points of this warp's next chunk
    auto load_chunk = [&](uint32_t c) {
        const uint64_t b = (uint64_t)c * kWChunk;
        const int2 *q = a.pts + b + lane;
        if (b + kWChunk <= a.n) {
#pragma unroll
            for (int j = 0; j < kWItems; ++j)
                pn[j] = __ldcs(q + 32 * j);
        } else {
#pragma unroll
            for (int j = 0; j < kWItems; ++j)
                pn[j] = c < nchunks && b + 32 * j + lane < a.n ? __ldcs(q + 32 * j) : make_int2(-1, -1);
        }
    };
    load_chunk(blockIdx.x * WARPS + warp);
    for (uint32_t ch = blockIdx.x * WARPS + warp; ch < nchunks; ch += nw) {
        const uint64_t base = (uint64_t)ch * kWChunk;
        if (lane == 0) { // the chunk after the next goes to L2; the next one to registers now
            const uint64_t nb = base + 2ull * nw * kWChunk;
            if (nb + kWChunk <= a.n)
                prefetch_l2_bulk(a.pts + nb, kWChunk * sizeof(int2));
        }
        int2 p[kWItems];
        uint32_t w[kWItems];
#pragma unroll
        for (int j = 0; j < kWItems; ++j)
            p[j] = pn[j];
        load_chunk(ch + nw);
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const uint32_t px = (uint32_t)p[j].x, py = (uint32_t)p[j].y;
            const bool ok = (px | py) < kBox; // both in [0, 2^30)
            const uint32_t sv = s_sum[(((py >> ix.ssh) << ix.sg) | (px >> ix.ssh)) & smask];
            w[j] = ok && sv != kSumEmpty ? (kCellInsideOne << 30) | sv : 0u;
            ld_idx_if<DISK>(w[j], ix.cell + (((py >> ix.sc) << ix.gc) | (px >> ix.sc)), keep, ok && sv == kSumMixed);
        }
#pragma unroll
        for (int j = 0; j < kWItems; ++j)
            if (!DISK && (w[j] >> 30) == kCellSub) // a disk index has one level
                w[j] = fine_word<false>(ix, w[j], (uint32_t)p[j].x, (uint32_t)p[j].y, keep);
        uint32_t bl[kWItems];
#pragma unroll
        for (int j = 0; j < kWItems; ++j)
            bl[j] = __ballot_sync(kFull, (int)w[j] < 0); // kCellList, kCellCoarseList
        if (lane == 0) {
            uint2 *d = reinterpret_cast<uint2 *>(pend + (uint64_t)ch * kWItems); // the bitmap is 8-byte aligned
#pragma unroll
            for (int j = 0; j < kWItems / 2; ++j)
                __stcg(d + j, make_uint2(bl[2 * j], bl[2 * j + 1]));
        }
        constexpr int kOne = int(kCellInsideOne << 30);
        // one: the polygon; list: its first entry (narrow: none; rewritten by pass
        // 1b); empty: none
        if (OUT == kOut16) {
            unsigned short *res = reinterpret_cast<unsigned short *>(a.res) + base + lane;
            if (base + kWChunk <= a.n) {
#pragma unroll
                for (int j = 0; j < kWItems; ++j)
                    __stcg(res + 32 * j, (unsigned short)((int)w[j] >= kOne ? w[j] : kRes16None));
            } else {
#pragma unroll
                for (int j = 0; j < kWItems; ++j)
                    if (base + 32 * j + lane < a.n)
                        __stcg(res + 32 * j, (unsigned short)((int)w[j] >= kOne ? w[j] : kRes16None));
            }
        } else if (OUT == kOut32) {
#pragma unroll
            for (int j = 0; j < kWItems; ++j)
                if (base + 32 * j + lane < a.n)
                    __stcg(a.res + base + 32 * j + lane, (w[j] >> 30) == kCellEmpty ? kResNone : w[j] & kPayloadMask);
        }
        uint32_t total = 0;
#pragma unroll
        for (int j = 0; j < kWItems; ++j)
            total += (int)w[j] >= kOne && in_bounds((w[j] & kPayloadMask) < ix.P, ix) ? 1u : 0u;
        if (hist) {
#pragma unroll
            for (int j = 0; j < kWItems; ++j)
                if ((int)w[j] >= kOne && in_bounds((w[j] & kPayloadMask) < ix.P, ix))
                    asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(hist_at + (w[j] << 2)) : "memory");
        } else if (a.counts) {
#pragma unroll
            for (int j = 0; j < kWItems; ++j)
                global_add_warp(a.counts, (int)w[j] >= kOne && in_bounds((w[j] & kPayloadMask) < ix.P, ix),
                                w[j] & kPayloadMask);
        }
        n_pairs += total;
        if (OUT != kOutCount) {
            total = __reduce_add_sync(kFull, total);
            if (lane == 0)
                a.tile_tot[ch] = total; // the chunk's total without its list points; pass 1b adds theirs
        }
    }
    if (hist) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < ix.P; i += kResolveSumThreads)
            if (s_hist[i])
                atomicAdd(a.counts + i, (unsigned long long)s_hist[i]);
    }
    add_stats(a.stats, 0u, 0u, 0u, n_pairs);
    if (blockIdx.x == 0 && threadIdx.x == 0)
        atomicAdd(a.stats + kStatPoints, (unsigned long long)a.n);
}

// With TMA, every warp stages its next chunk's points in its own shared-memory
// buffer with one bulk copy, issued as soon as it has read the current chunk
// from there: the points arrive while the chunk is resolved, and their loads
// cost the L1 nothing.  A warp's last chunk, when it is not full, is loaded
// with plain loads.
//
// Without the summary.
template <int THREADS, bool TMA, int OUT, bool DISK>
__global__ void __launch_bounds__(THREADS, TMA ? 6 : kResolveMinBlocks)
    k_resolve(const __grid_constant__ JoinLaunch a, uint32_t *pend, uint32_t nchunks, int use_hist)
{
    constexpr int WARPS = THREADS / 32;
    extern __shared__ __align__(16) unsigned char s_raw[];
    const IndexView &ix = a.ix;
    int2 *s_buf = reinterpret_cast<int2 *>(s_raw) + (size_t)(threadIdx.x >> 5) * kWChunk;
    uint64_t *s_bar = reinterpret_cast<uint64_t *>(s_raw + size_t(WARPS) * kWChunk * sizeof(int2)) +
                      (threadIdx.x >> 5);
    uint32_t *s_hist = reinterpret_cast<uint32_t *>(s_raw + resolve_smem_head(WARPS, false, 0, TMA));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t keep = policy_evict_last();
    const bool hist = use_hist && a.counts;
    const uint32_t nw = gridDim.x * WARPS;
    auto full = [&](uint32_t c) { return (uint64_t)(c + 1) * kWChunk <= a.n; };
    if constexpr (TMA) {
        const uint32_t c0 = blockIdx.x * WARPS + warp;
        if (lane == 0) {
            mbar_init(s_bar, 1);
            if (c0 < nchunks && full(c0))
                bulk_load(s_buf, a.pts + (uint64_t)c0 * kWChunk, kWChunk * sizeof(int2), s_bar);
        }
    }
    if (hist)
        for (uint32_t i = threadIdx.x; i < ix.P; i += THREADS)
            s_hist[i] = 0;
    __syncthreads();
    uint32_t n_pts = 0, n_pairs = 0, phase = 0;
    for (uint32_t ch = blockIdx.x * WARPS + warp; ch < nchunks; ch += nw) {
        const uint64_t base = (uint64_t)ch * kWChunk;
        const uint32_t npts = (uint32_t)min((uint64_t)kWChunk, a.n - base);
        const int2 *pts = a.pts + base;
        uint32_t *res = a.res + base;
        uint16_t *res16 = reinterpret_cast<uint16_t *>(a.res) + base;
        int2 p[kWItems];
        uint32_t w[kWItems];
        if (TMA && npts == kWChunk) {
            if (!mbar_wait(s_bar, phase, kWaitTries)) {
                // the copy did not arrive: report it, give it one more bounded wait, stop
                if (lane == 0)
                    atomicOr(a.err, kErrTimeout);
                mbar_wait(s_bar, phase, kWaitTries);
                break;
            }
            phase ^= 1u;
#pragma unroll
            for (int j = 0; j < kWItems; ++j)
                p[j] = s_buf[j * 32 + lane];
            __syncwarp();
            const uint32_t nx = ch + nw;
            if (lane == 0 && nx < nchunks && full(nx))
                bulk_load(s_buf, a.pts + (uint64_t)nx * kWChunk, kWChunk * sizeof(int2), s_bar);
        } else {
            if (!TMA && kPrefetchChunks > 0 && lane == 0) { // (with TMA only a ragged last chunk comes here)
                // this warp's chunk kPrefetchChunks ahead goes to L2 while this one is resolved
                const uint64_t nb = base + (uint64_t)kPrefetchChunks * nw * kWChunk;
                if (nb + kWChunk <= a.n)
                    prefetch_l2_bulk(a.pts + nb, kWChunk * sizeof(int2));
            }
#pragma unroll
            for (int j = 0; j < kWItems; ++j) {
                const uint32_t loc = j * 32 + lane;
                p[j] = loc < npts ? __ldcs(pts + loc) : make_int2(-1, -1);
            }
        }
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            // x, y >= 0 and both < 2^30 iff their bitwise or is below 2^30
            const bool ok = (uint32_t)(p[j].x | p[j].y) < kBox;
            const uint32_t px = ok ? (uint32_t)p[j].x : 0u, py = ok ? (uint32_t)p[j].y : 0u;
            w[j] = 0u;
            if (ok)
                w[j] = coarse_word<DISK>(ix, px, py, keep);
        }
#pragma unroll
        for (int j = 0; j < kWItems; ++j)
            if (!DISK && (w[j] >> 30) == kCellSub) // a disk index has one level
                w[j] = fine_word<false>(ix, w[j], (uint32_t)p[j].x, (uint32_t)p[j].y, keep);
        uint32_t total = 0, mask = 0;
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const uint32_t kind = w[j] >> 30, loc = j * 32 + lane, pay = w[j] & kPayloadMask;
            const bool one = kind == kCellInsideOne && in_bounds(pay < ix.P, ix);
            total += one ? 1u : 0u;
            if (a.counts) {
                if (!hist)
                    global_add_warp(a.counts, one, pay);
                else if (one)
                    atomicAdd(s_hist + pay, 1u);
            }
            // one: the polygon; list: its first entry (narrow: none; rewritten
            // by pass 1b); empty: none
            if (OUT != kOutCount && loc < npts) {
                if (OUT == kOut16)
                    __stcg(reinterpret_cast<unsigned short *>(res16 + loc),
                           (unsigned short)(kind == kCellInsideOne ? pay : kRes16None));
                else
                    __stcg(res + loc, kind == kCellEmpty ? kResNone : pay);
            }
            const uint32_t bl = __ballot_sync(kFull, kind >= kCellList); // or kCellCoarseList
            mask = lane == j ? bl : mask;
        }
        if (lane < kWItems)
            __stcg(pend + (uint64_t)ch * kWItems + lane, mask);
        n_pts += lane == 0 ? npts : 0u;
        n_pairs += total;
        if (OUT == kOutCount)
            continue;
        total = warp_sum32(total);
        if (lane == 0)
            a.tile_tot[ch] = total; // the chunk's total without its list points; pass 1b adds theirs
    }
    if (hist) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < ix.P; i += THREADS)
            if (s_hist[i])
                atomicAdd(a.counts + i, (unsigned long long)s_hist[i]);
    }
    add_stats(a.stats, n_pts, 0u, 0u, n_pairs);
}

// Pass 1b.  Up to kSmallHist polygons are counted in shared memory: where many points lie
// in several polygons (overlapping queries) a global atomic per hit on a few
// hundred counters was what this pass waited for (20M points x 256 buffered
// queries: 1545 -> 185 us).
constexpr uint32_t kSmallHist = 2048;

// The rows go through two queues of the warp.  Rows are resolved kWalkBatch rounds
// of 32 at a time (their points, then their coarse words, then their fine words:
// three round trips for 128 rows instead of for 32), and those with a list are
// walked 32 at a time (500M points x 256 queries 4.54 -> 4.39 ms at 72 registers and
// three CTAs per SM; with local edge lists 2.7 ms at 64 registers and four).
//
// With ALL (the count aggregate over a cell directory) a marked row is any row
// of a mixed coarse cell: rows that its fine cell resolves are counted here.
template <bool FP32, int OUT, int KIND, bool ALL>
__global__ void __launch_bounds__(kThreads, KIND == kNear ? 3 : kWalkMinBlocks) k_walk(const __grid_constant__ JoinLaunch a, uint32_t *pend,
                                                                   uint32_t nwords, int group_log2)
{
    static_assert(!ALL || OUT == kOutCount, "ALL keeps nothing per row");
    constexpr bool L1 = ALL || KIND == kDisk; // index words
    const int gl = ALL || OUT == kOut32 ? group_log2 : 5; // see launch_walk
    __shared__ uint32_t s_qa[kWarps * kWalkQueue];
    __shared__ uint4 s_la[kWarps * kWalkQueue];
    __shared__ uint32_t s_pa[kWarps * kWaveWords];
    __shared__ uint32_t s_hist[kSmallHist];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *s_q = s_qa + warp * kWalkQueue; // rows to resolve
    uint4 *s_l = s_la + warp * kWalkQueue;    // (x, y, first entry, row) to walk
    uint32_t *s_par = s_pa + warp * kWaveWords;
    const IndexView &ix = a.ix;
    const uint64_t keep = policy_evict_last();
    const bool hist = a.counts && ix.P <= kSmallHist;
    if (hist) {
        for (uint32_t i = threadIdx.x; i < ix.P; i += kThreads)
            s_hist[i] = 0;
        __syncthreads();
    }
    uint32_t n_tests = 0, n_esc = 0, n_pairs = 0, n_pts = 0, qn = 0, ln = 0;
    // ALL: neighbouring rows mostly share a polygon (a clustered table): one
    // atomic per distinct polygon of the warp
    auto count_warp = [&](bool has, uint32_t q) {
        if (hist)
            hist_add_warp(s_hist, has, q);
        else
            global_add_warp(a.counts, has, q);
    };
    // walks the last m <= 32 queued lists, one per lane
    auto walk = [&](uint32_t m) {
        const bool has = (uint32_t)lane < m;
        const uint4 it = s_l[ln - m + (has ? lane : 0)]; // idle lanes walk nothing
        ln -= m;
        const uint32_t row = it.w;
        uint32_t f = 0, c = 0;
        uint64_t ids = 0; // kOut16 and a.aux: the first polygons, aux_bits each
        walk_list_wave<FP32, KIND>(ix, has, it.z, (int)it.x, (int)it.y, n_tests, n_esc, keep, s_par, [&](uint32_t q) {
            if (OUT == kOut16 && a.aux && (c + 1) * a.aux_bits <= 64)
                ids |= (uint64_t)q << (a.aux_bits * c);
            f = c ? f : q;
            ++c;
            if (a.counts && !(ALL && c == 1))
                hist ? (void)atomicAdd(s_hist + q, 1u) : (void)atomicAdd(a.counts + q, 1ull);
        }, &a.near);
        if (ALL)
            count_warp(c >= 1, f);
        n_pairs += c;
        if (OUT != kOutCount && has) {
            if (OUT == kOut16) {
                __stcg(reinterpret_cast<unsigned short *>(a.res) + row,
                       (unsigned short)(c == 0 ? kRes16None : c == 1 ? f : c));
                // the row's bit stays set iff the point is in several polygons;
                // only this warp reads or writes the bitmap words of its range
                if (c < 2)
                    atomicAnd(pend + (row >> 5), ~(1u << (row & 31)));
                else if (a.aux && c * a.aux_bits <= 64)
                    __stcg(reinterpret_cast<unsigned long long *>(a.aux) + row, (unsigned long long)ids);
            } else {
                __stcg(a.res + row, res_encode(c, f));
            }
            if (c)
                atomicAdd(a.tile_tot + row / kWChunk, (unsigned long long)c);
        }
        __syncwarp(); // the queue is rewritten after the round
    };
    // resolves the last m <= 32 B queued rows, B per lane, and walks what fills rounds
    constexpr int B = kWalkBatch;
    auto take = [&](uint32_t m) {
        __syncwarp();
        qn -= m;
        uint32_t row[B], w[B];
        int2 p[B];
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const uint32_t k = u * 32 + lane;
            row[u] = s_q[qn + (k < m ? k : 0)]; // idle lanes repeat the first row and add nothing
            p[u] = a.pts[row[u]];
        }
        // the list's first entry: stored by pass 1a (32-bit results), else the
        // cell resolved again; a marked row's point is in the box
#pragma unroll
        for (int u = 0; u < B; ++u)
            w[u] = OUT == kOut32 ? (kCellList << 30) | __ldcg(a.res + row[u])
                                 : coarse_word<L1>(ix, (uint32_t)p[u].x, (uint32_t)p[u].y, keep);
        if (OUT != kOut32) {
#pragma unroll
            for (int u = 0; u < B; ++u)
                if (KIND != kDisk && (w[u] >> 30) == kCellSub)
                    w[u] = fine_word<L1>(ix, w[u], (uint32_t)p[u].x, (uint32_t)p[u].y, keep);
        }
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const bool has = u * 32 + lane < m;
            const uint32_t kind = w[u] >> 30, pay = w[u] & kPayloadMask;
            const bool lst = has && kind >= kCellList;
            if (ALL) {
                const bool one = has && kind == kCellInsideOne && in_bounds(pay < ix.P, ix);
                count_warp(one, pay);
                n_pairs += one ? 1u : 0u;
            } else {
                in_bounds(!has || lst, ix);
            }
            const uint32_t bl = __ballot_sync(kFull, lst);
            if (lst)
                s_l[ln + __popc(bl & lanemask_lt())] = make_uint4((uint32_t)p[u].x, (uint32_t)p[u].y, pay, row[u]);
            ln += __popc(bl);
        }
        __syncwarp();
        while (ln >= 32)
            walk(32);
    };
    // this warp's words: every nw-th group of 2^gl (at most 32), so that a run of marked
    // rows (a clustered table) is shared out; a lane per word, BW groups loaded ahead
    constexpr int BW = 4;
    const uint64_t nw = (uint64_t)gridDim.x * kWarps, g0 = (uint64_t)blockIdx.x * kWarps + warp;
    auto load = [&](uint64_t g) {
        const uint64_t i = (g << gl) + lane;
        return lane < 1 << gl && i < nwords ? __ldcs(pend + i) : 0u;
    };
    uint32_t nxt[BW];
#pragma unroll
    for (int k = 0; k < BW; ++k)
        nxt[k] = load(g0 + k * nw);
    for (uint64_t g = g0; (g << gl) < nwords; g += BW * nw) {
        uint32_t cur[BW];
#pragma unroll
        for (int k = 0; k < BW; ++k) {
            cur[k] = nxt[k];
            nxt[k] = load(g + (BW + k) * nw);
        }
#pragma unroll 1
        for (int k = 0; k < BW; ++k) { // not unrolled: one copy of the walk
            const uint64_t wi = ((g + k * nw) << gl) + lane;
            uint32_t m = cur[0];
#pragma unroll
            for (int t = 0; t + 1 < BW; ++t)
                cur[t] = cur[t + 1];
            if (ALL) {
                // marked rows come in runs: a lane per row of a word, so that a round's
                // points, cells and lists are mostly the same (a row of each lane's word at
                // a time: 500M points x 40000 cells 1389 us, now 1219)
                n_pts += __popc(m);
                for (uint32_t todo = __ballot_sync(kFull, m != 0); todo; todo &= todo - 1) {
                    const int src = __ffs(todo) - 1;
                    const uint32_t word = __shfl_sync(kFull, m, src);
                    const uint32_t row = (uint32_t)((wi - lane + src) * 32) + lane;
                    if ((word >> lane) & 1u) {
                        s_q[qn + __popc(word & lanemask_lt())] = row;
                        prefetch_l2(a.pts + row);
                    }
                    qn += __popc(word);
                    if (qn >= 32 * B)
                        take(32 * B);
                }
                continue;
            }
            while (__any_sync(kFull, m != 0)) {
                const bool has = m != 0;
                const uint32_t b = (uint32_t)__ffs(m) - 1u;
                m &= m - 1u;
                const uint32_t bl = __ballot_sync(kFull, has);
                if (has) {
                    const uint32_t row = (uint32_t)(wi * 32 + b);
                    s_q[qn + __popc(bl & lanemask_lt())] = row;
                    prefetch_l2(a.pts + row); // loaded when its round is resolved
                }
                qn += __popc(bl);
                if (qn >= 32 * B)
                    take(32 * B);
            }
        }
    }
    if (qn)
        take(qn);
    if (ln)
        walk(ln);
    if (hist) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < ix.P; i += kThreads)
            if (s_hist[i])
                atomicAdd(a.counts + i, (unsigned long long)s_hist[i]);
    }
    add_stats(a.stats, n_pts, n_tests, n_esc, n_pairs);
}

// Opt a kernel in to the shared memory it needs (once per device).
template <class K>
cudaError_t smem_opt_in(K kernel, size_t bytes, bool (&done)[64])
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 64 && done[dev])
        return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
    if (e == cudaSuccess && dev < 64)
        done[dev] = true;
    return e;
}

template <bool FP32, int OUT, int KIND, bool ALL = false>
cudaError_t launch_walk(const JoinLaunch &a, uint32_t *pend, cudaStream_t s)
{
    // Groups of fewer words where the marked rows lie close together: a warp goes through
    // its own one round after the other.  Over a clustered table (ALL) they come in runs,
    // and a warp per 1024 rows left most warps without any: 32 groups a warp where the
    // table has the words (300k points x 120 overlapping queries 310 -> 105 us, 20M
    // 1437 -> 463; 20M x 300 cells 114 -> 114; 500M x 40000 cells takes whole groups).
    // With wide results, one (300k points x 70000 buffered squares 88 -> 62 us, 1.5M 170 ->
    // 146).  Rows of narrow results are spread thin, and a smaller group would only
    // leave rounds part empty (1.5M x 300 cells 35 -> 37).
    // a warp per group of 32 words, shared out by stride over what the chip holds
    // at once (1M points: 61 warps of 512 words took 20.3 us, 977 of 32 take 7.5;
    // 100M x 2000 cells: 1.8 waves 87 us, one 74), or over up to six times as many
    // while a warp keeps kWalkGroups groups, which evens out long walks (500M x 256
    // queries: one wave 3.15 ms, six 2.95)
    const uint64_t nwords = (a.n + kWChunk - 1) / kWChunk * kWItems;
    auto kern = k_walk<FP32, OUT, KIND, ALL>;
    const uint32_t wave = (uint32_t)persistent_grid(kern, kThreads, 0, UINT32_MAX);
    int gl = 5;
    if (ALL || OUT == kOut32)
        while (gl && (nwords >> gl) < (uint64_t)wave * kWarps * (ALL ? 32 : 1))
            --gl;
    const uint32_t nblk = uint32_t((nwords + (kWarps << gl) - 1) / (kWarps << gl));
    const uint32_t waves = std::min(std::max(nblk / (wave * kWalkGroups), 1u), 6u);
    kern<<<std::min(nblk, wave * waves), kThreads, 0, s>>>(a, pend, uint32_t(nwords), gl);
    return cudaGetLastError();
}

// Pass 1 of a small table in one launch: a warp per 256-point chunk resolves its
// points as pass 1a does and walks its own list points at once.  A table of up
// to kSmallChunks chunks is bound by launches and by chains of dependent loads,
// not by bandwidth, and the persistent CTAs of pass 1a would copy the 128 KB
// summary for a few chunks each.  CTA of kThreads, no barrier between its warps
// but for the counters (a CTA's points counted in shared memory when P is at
// most kSmallHist).  Whole join with k_wemit16<SELF>, against pass 1a + 1b + scan
// + pass 3, 2000-cell map: 20k points 19.1 against 30.9 us, 500k 21.2 / 32.9, 1M
// 26.7 / 35.9, 1.5M 39.3 / 41.1, 2M 48.5 / 41.1, 3M 71.0 / 51.5; 256 stars: 1M 24.1 /
// 32.9, 2M 35.1 / 35.0.  The two cross between 1.5M and 2M points.  The line is
// below that, at 1M, where an earlier form of this kernel had it.
constexpr uint32_t kSmallChunks = 4096;

template <bool FP32, int OUT, int KIND>
__global__ void __launch_bounds__(kThreads, KIND == kNear ? 3 : 4) k_small(const __grid_constant__ JoinLaunch a, uint32_t *pend,
                                                       uint32_t nchunks, int use_hist)
{
    __shared__ uint4 s_qa[kWarps * kWChunk]; // (x, y, first entry, row in the chunk)
    __shared__ uint32_t s_pa[kWarps * kWaveWords];
    __shared__ uint32_t s_ma[kWarps * kWItems]; // rows in several polygons
    __shared__ uint32_t s_hist[kSmallHist];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint4 *s_q = s_qa + warp * kWChunk;
    uint32_t *s_m = s_ma + warp * kWItems;
    const IndexView &ix = a.ix;
    const uint64_t keep = policy_evict_last();
    const bool hist = use_hist && a.counts;
    uint32_t n_tests = 0, n_esc = 0, total = 0, npts = 0;
    if (hist) {
        for (uint32_t i = threadIdx.x; i < ix.P; i += kThreads)
            s_hist[i] = 0;
        __syncthreads();
    }
    auto count1 = [&](bool has, uint32_t q) {
        if (has && a.counts)
            hist ? (void)atomicAdd(s_hist + q, 1u) : (void)atomicAdd(a.counts + q, 1ull);
    };
    const uint32_t ch = blockIdx.x * kWarps + warp;
    if (ch < nchunks) {
        const uint64_t base = (uint64_t)ch * kWChunk;
        npts = (uint32_t)min((uint64_t)kWChunk, a.n - base);
        unsigned short *res16 = reinterpret_cast<unsigned short *>(a.res) + base;
        int2 p[kWItems];
        uint32_t w[kWItems];
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const uint32_t loc = j * 32 + lane;
            p[j] = loc < npts ? __ldcs(a.pts + base + loc) : make_int2(-1, -1);
        }
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            w[j] = 0u;
            if ((uint32_t)(p[j].x | p[j].y) < kBox)
                w[j] = coarse_word<KIND == kDisk>(ix, (uint32_t)p[j].x, (uint32_t)p[j].y, keep);
        }
#pragma unroll
        for (int j = 0; j < kWItems; ++j)
            if (KIND != kDisk && (w[j] >> 30) == kCellSub)
                w[j] = fine_word<false>(ix, w[j], (uint32_t)p[j].x, (uint32_t)p[j].y, keep);
        if (lane < kWItems)
            s_m[lane] = 0u;
        uint32_t qn = 0;
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const uint32_t kind = w[j] >> 30, loc = j * 32 + lane, pay = w[j] & kPayloadMask;
            const bool one = kind == kCellInsideOne && in_bounds(pay < ix.P, ix), lst = kind >= kCellList;
            total += one ? 1u : 0u;
            count1(one, pay);
            if (OUT == kOut16 && loc < npts && !lst)
                __stcg(res16 + loc, (unsigned short)(one ? pay : kRes16None));
            const uint32_t bl = __ballot_sync(kFull, lst);
            if (lst)
                s_q[qn + __popc(bl & lanemask_lt())] = make_uint4((uint32_t)p[j].x, (uint32_t)p[j].y, pay, loc);
            qn += __popc(bl);
        }
        __syncwarp();
        for (uint32_t k0 = 0; k0 < qn; k0 += 32) {
            const bool has = k0 + lane < qn;
            const uint4 it = s_q[has ? k0 + lane : k0]; // idle lanes walk nothing
            uint32_t f = 0, c = 0;
            uint64_t ids = 0; // kOut16 and a.aux: the first polygons, aux_bits each
            walk_list_wave<FP32, KIND>(ix, has, it.z, (int)it.x, (int)it.y, n_tests, n_esc, keep, s_pa + warp * kWaveWords,
                                 [&](uint32_t q) {
                                     if (OUT == kOut16 && a.aux && (c + 1) * a.aux_bits <= 64)
                                         ids |= (uint64_t)q << (a.aux_bits * c);
                                     f = c ? f : q;
                                     ++c;
                                     count1(true, q);
                                 }, &a.near);
            total += c;
            if (OUT == kOut16 && has) {
                __stcg(res16 + it.w, (unsigned short)(c == 0 ? kRes16None : c == 1 ? f : c));
                if (c >= 2) {
                    atomicOr(s_m + (it.w >> 5), 1u << (it.w & 31));
                    if (a.aux && c * a.aux_bits <= 64)
                        __stcg(reinterpret_cast<unsigned long long *>(a.aux) + base + it.w, (unsigned long long)ids);
                }
            }
        }
        __syncwarp();
        if (OUT != kOutCount) {
            if (lane < kWItems)
                __stcg(pend + (uint64_t)ch * kWItems + lane, s_m[lane]);
            const uint32_t t = warp_sum32(total);
            if (lane == 0)
                a.tile_tot[ch] = t;
        }
    }
    if (hist) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < ix.P; i += kThreads)
            if (s_hist[i])
                atomicAdd(a.counts + i, (unsigned long long)s_hist[i]);
    }
    add_stats(a.stats, lane == 0 ? npts : 0u, n_tests, n_esc, total);
}

// Pass 1 of a disk index in one kernel: joins of more than kDiskSplit disks, and the
// counts but those of large tables in row order (use_split_count).  Disk lists are short
// and their tests cheap: a lane walks its own list as soon as a round of 32 list points
// is queued (across chunks), with the point at hand.  A point in a block that no disk
// reaches leaves by the cover bitmap, in shared memory (8 KB where the summary takes 128,
// so four CTAs per SM keep 32 warps).  Counts in shared memory up to kHistMax disks.
// Against passes 1a and 1b, which re-read their rows: counts over a clustered table, 20M
// points x 64 / 1024 / 4096 disks 50 / 59 / 73 us against 61 / 96 / 158, of 300k x 1024
// 12.1 against 14.5.  Joins: 100M x 1024 disks 500 us against 433, 20M x 1024 125 against
// 117; 20M x 4096, which k_walk counts in global memory, 140 against 185, x 20000 159
// against 198, and with 90 % of 20M points in 512 of 4096 disks, where counters take
// millions of hits each, 6.8 ms against 59.6.
constexpr uint32_t kDiskSplit = kSmallHist;
constexpr uint32_t kDiskCoverWords = 1u << (2 * kCoverLog2 - 5);
constexpr int kDiskQueue = kWChunk + 32; // a chunk's points plus a partial round
constexpr size_t kDiskSmem = size_t(kWarps) * kDiskQueue * sizeof(uint4) + kDiskCoverWords * sizeof(uint32_t);

template <int OUT>
__global__ void __launch_bounds__(kThreads, 4)
    k_disk_pass1(const __grid_constant__ JoinLaunch a, uint32_t *pend, uint32_t nchunks, int use_hist)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint4 *s_q = reinterpret_cast<uint4 *>(s_raw) + warp * kDiskQueue; // (x, y, list, row)
    uint32_t *s_cov = reinterpret_cast<uint32_t *>(s_raw + size_t(kWarps) * kDiskQueue * sizeof(uint4));
    uint32_t *s_hist = s_cov + kDiskCoverWords;
    const IndexView &ix = a.ix;
    const uint64_t keep = policy_evict_last();
    const bool hist = use_hist && a.counts;
    for (uint32_t i = threadIdx.x; i < max(1u, (1u << (2 * ix.cg)) >> 5); i += kThreads)
        s_cov[i] = __ldg(ix.cover + i);
    if (hist)
        for (uint32_t i = threadIdx.x; i < ix.P; i += kThreads)
            s_hist[i] = 0;
    __syncthreads();
    auto count1 = [&](bool has, uint32_t q) { // one disk for every lane with has (converged warp)
        if (!a.counts)
            return;
        if (!hist)
            global_add_warp(a.counts, has, q);
        else if (has)
            atomicAdd(s_hist + q, 1u);
    };
    unsigned short *res16 = reinterpret_cast<unsigned short *>(a.res);
    uint32_t n_tests = 0, n_pts = 0, n_pairs = 0, qn = 0; // qn: queued points, < 32 between chunks
    auto walk = [&](uint32_t k0, uint32_t m) { // queued points [k0, k0 + m), m <= 32
        const bool has = (uint32_t)lane < m;
        const uint4 it = s_q[k0 + (has ? lane : 0)]; // idle lanes repeat lane 0's walk, uncounted
        const uint32_t *e = a.near.dent + it.z;
        const uint32_t n = ld_idx(e, keep);
        uint32_t c = 0, f = 0, tests = 0;
        uint64_t ids = 0; // kOut16 and a.aux: the first disks, aux_bits each
        for (uint32_t k = 1; k <= n; ++k) {
            const uint32_t en = ld_idx(e + k, keep), q = en >> 1;
            bool in = true;
            if (en & 1u) {
                ++tests;
                in = in_disk(__ldg(a.near.disk + q), (int)it.x, (int)it.y);
            }
            if (in) {
                if (OUT == kOut16 && a.aux && (c + 1) * a.aux_bits <= 64)
                    ids |= (uint64_t)q << (a.aux_bits * c);
                if (!c)
                    f = q; // counted with the warp below
                else if (has && a.counts)
                    hist ? (void)atomicAdd(s_hist + q, 1u) : (void)atomicAdd(a.counts + q, 1ull);
                ++c;
            }
        }
        c = has ? c : 0u;
        n_tests += has ? tests : 0u;
        n_pairs += c;
        __syncwarp();
        count1(c >= 1, f);
        if (OUT != kOutCount && has) {
            const uint32_t row = it.w;
            if (OUT == kOut16) {
                __stcg(res16 + row, (unsigned short)(c == 0 ? kRes16None : c == 1 ? f : c));
                if (c >= 2) { // the row's bit: only this warp writes the words of its chunks
                    atomicOr(pend + (row >> 5), 1u << (row & 31));
                    if (a.aux && c * a.aux_bits <= 64)
                        __stcg(reinterpret_cast<unsigned long long *>(a.aux) + row, (unsigned long long)ids);
                }
            } else {
                __stcg(a.res + row, res_encode(c, f));
            }
            if (c)
                atomicAdd(a.tile_tot + row / kWChunk, (unsigned long long)c);
        }
        __syncwarp();
    };
    const uint32_t nw = gridDim.x * kWarps;
    for (uint32_t ch = blockIdx.x * kWarps + warp; ch < nchunks; ch += nw) {
        const uint64_t base = (uint64_t)ch * kWChunk;
        const uint32_t npts = (uint32_t)min((uint64_t)kWChunk, a.n - base);
        n_pts += lane == 0 ? npts : 0u;
        int2 p[kWItems];
        uint32_t w[kWItems];
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const uint32_t loc = j * 32 + lane;
            p[j] = loc < npts ? __ldcs(a.pts + base + loc) : make_int2(-1, -1);
        }
        if (OUT == kOut16 && lane < kWItems)
            __stcg(pend + (uint64_t)ch * kWItems + lane, 0u);
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const uint32_t px = (uint32_t)p[j].x, py = (uint32_t)p[j].y;
            const uint32_t b = (((py & (kBox - 1)) >> ix.scv) << ix.cg) | ((px & (kBox - 1)) >> ix.scv);
            const bool ok = (px | py) < kBox && ((s_cov[b >> 5] >> (b & 31)) & 1u);
            w[j] = ok ? ld_idx(ix.cell + ((((py & (kBox - 1)) >> ix.sc) << ix.gc) | ((px & (kBox - 1)) >> ix.sc)), keep) : 0u;
        }
        uint32_t total = 0;
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const uint32_t kind = w[j] >> 30, loc = j * 32 + lane, pay = w[j] & kPayloadMask;
            const bool one = kind == kCellInsideOne && in_bounds(pay < ix.P, ix), lst = kind >= kCellList;
            total += one ? 1u : 0u;
            count1(one, pay);
            if (OUT != kOutCount && loc < npts && !lst) {
                if (OUT == kOut16)
                    __stcg(res16 + base + loc, (unsigned short)(one ? pay : kRes16None));
                else
                    __stcg(a.res + base + loc, one ? pay : kResNone);
            }
            const uint32_t bl = __ballot_sync(kFull, lst);
            if (lst)
                s_q[qn + __popc(bl & lanemask_lt())] =
                    make_uint4((uint32_t)p[j].x, (uint32_t)p[j].y, pay, (uint32_t)(base + loc));
            qn += __popc(bl);
        }
        n_pairs += total;
        if (OUT != kOutCount) {
            total = __reduce_add_sync(kFull, total);
            if (lane == 0)
                a.tile_tot[ch] = total; // without its queued points, which add theirs
        }
        __syncwarp();
        if (qn >= 32) {
            uint32_t k0 = 0;
            for (; qn - k0 >= 32; k0 += 32)
                walk(k0, 32);
            const uint32_t rem = qn - k0; // the partial round (< 32, from k0 >= 32) to the front
            const uint4 it = (uint32_t)lane < rem ? s_q[k0 + lane] : make_uint4(0u, 0u, 0u, 0u);
            __syncwarp();
            if ((uint32_t)lane < rem)
                s_q[lane] = it;
            qn = rem;
            __syncwarp();
        }
    }
    if (qn)
        walk(0, qn);
    if (hist) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < ix.P; i += kThreads)
            if (s_hist[i])
                atomicAdd(a.counts + i, (unsigned long long)s_hist[i]);
    }
    add_stats(a.stats, n_pts, n_tests, 0u, n_pairs);
}

template <int OUT>
cudaError_t launch_disk_pass1(const JoinLaunch &a, uint32_t *pend, cudaStream_t s)
{
    static bool done[64] = {};
    if (a.n >= (1ull << 32))
        return cudaErrorInvalidValue; // rows are 32-bit
    const uint64_t nchunks = (a.n + kWChunk - 1) / kWChunk;
    const int use_hist = a.counts && a.ix.P <= (uint32_t)kHistMax ? 1 : 0;
    const size_t smem = kDiskSmem + (use_hist ? sizeof(uint32_t) * a.ix.P : 0);
    auto kern = k_disk_pass1<OUT>;
    const cudaError_t e = smem_opt_in(kern, kDiskSmem + sizeof(uint32_t) * kHistMax, done);
    if (e != cudaSuccess)
        return e;
    const uint32_t nblk = uint32_t((nchunks + kWarps - 1) / kWarps);
    kern<<<persistent_grid(kern, kThreads, smem, nblk), kThreads, smem, s>>>(a, pend, uint32_t(nchunks), use_hist);
    return cudaGetLastError();
}

// Pass 3 of the join with warp chunks: every warp writes the pairs of its
// chunks from the stored per-point results at the chunk's scanned offset.
// Lane order within a round of 32 points, rounds in order: point order.  A
// point in one polygon is written at once; a point in several is queued (its
// row and its offset; its count comes with its stored result), and the warp
// walks its queue 32 points at a time afterwards (all lanes busy, as in pass
// 1), loading the queued points' coordinates then, one independent load per
// lane, to write their pairs.
constexpr size_t kEmitSmem = size_t(kWarps) * kWChunk * (sizeof(uint32_t) + sizeof(unsigned long long)) +
                             size_t(kWarps) * kWaveWords * sizeof(uint32_t);

// (k_wemit: 32-bit results, more than kRes16MaxP polygons.)
template <bool FP32, int KIND>
__global__ void __launch_bounds__(kThreads, 3) k_wemit(const __grid_constant__ JoinLaunch a, const unsigned long long *chunk_off,
                                                       uint32_t nchunks)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long *s_o = reinterpret_cast<unsigned long long *>(s_raw) + warp * kWChunk;
    uint32_t *s_q = reinterpret_cast<uint32_t *>(s_raw + size_t(kWarps) * kWChunk * sizeof(unsigned long long)) +
                    warp * kWChunk; // rows within the chunk
    uint32_t *s_par = reinterpret_cast<uint32_t *>(s_raw + size_t(kWarps) * kWChunk *
                                                               (sizeof(unsigned long long) + sizeof(uint32_t))) +
                      warp * kWaveWords; // words of walk_list_wave
    const uint64_t keep = policy_evict_last();
    const uint32_t nw = gridDim.x * kWarps;
    for (uint32_t ch = blockIdx.x * kWarps + warp; ch < nchunks; ch += nw) {
        const uint64_t base = (uint64_t)ch * kWChunk;
        const uint32_t npts = (uint32_t)min((uint64_t)kWChunk, a.n - base);
        unsigned long long run = chunk_off[ch] + (a.pair_base ? *a.pair_base : 0ull);
        uint32_t res[kWItems];
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const uint32_t loc = j * 32 + lane;
            res[j] = loc < npts ? __ldcs(a.res + base + loc) : kResNone;
        }
        uint32_t qn = 0;
#pragma unroll
        for (int j = 0; j < kWItems; ++j) {
            const uint32_t loc = j * 32 + lane;
            const uint32_t r = res[j], pid = a.pid0 + (uint32_t)(base + loc);
            const bool multi = r != kResNone && (r & kResMulti);
            uint32_t c = r == kResNone ? 0u : 1u, pre, tot;
            if (!__any_sync(kFull, multi)) {
                const uint32_t bl = __ballot_sync(kFull, c != 0);
                pre = __popc(bl & lanemask_lt());
                tot = __popc(bl);
            } else {
                if (multi) {
                    if (r & kResCount) {
                        c = (r >> 20) & 0x3ffu;
                    } else { // count not stored: count again
                        const int2 p = a.pts[base + loc];
                        uint32_t f = 0, t = 0, e = 0;
                        c = KIND == kPoly   ? point_count<FP32>(a.ix, p.x, p.y, f, t, e, keep)
                            : KIND == kNear ? near_count<FP32>(a.ix, a.near, p.x, p.y, keep)
                                            : disk_count(a.ix, a.near, p.x, p.y, keep);
                    }
                }
                uint32_t inc = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t v = __shfl_up_sync(kFull, inc, o);
                    if (lane >= o)
                        inc += v;
                }
                pre = inc - c;
                tot = __shfl_sync(kFull, inc, 31);
                const uint32_t bl = __ballot_sync(kFull, multi);
                if (multi) {
                    const uint32_t slot = qn + __popc(bl & lanemask_lt());
                    s_q[slot] = loc;
                    s_o[slot] = run + pre;
                    c = 0; // written from the queue
                }
                qn += __popc(bl);
            }
            if (c) {
                const unsigned long long o = run + pre;
                if (o < a.cap)
                    __stcs(a.pairs + o, make_uint2(pid, r));
            }
            run += tot;
        }
        __syncwarp();
        for (uint32_t k0 = 0; k0 < qn; k0 += 32) {
            // the whole warp walks the queued points' lists together
            const bool has = k0 + lane < qn;
            const uint32_t loc = has ? s_q[k0 + lane] : 0u;
            unsigned long long o = has ? s_o[k0 + lane] : 0ull;
            const int2 p = has ? a.pts[base + loc] : make_int2(0, 0);
            const uint32_t pid = a.pid0 + (uint32_t)(base + loc);
            const uint32_t w = has ? resolve<KIND, KIND == kDisk>(a.ix, (uint32_t)p.x, (uint32_t)p.y, keep) : 0u;
            uint32_t t = 0, e = 0;
            walk_list_wave<FP32, KIND>(a.ix, (w >> 30) >= kCellList, w & kPayloadMask, p.x, p.y, t, e, keep, s_par,
                                 [&](uint32_t q) {
                                     if (o < a.cap)
                                         __stcs(a.pairs + o, make_uint2(pid, q));
                                     ++o;
                                 }, &a.near);
        }
        __syncwarp(); // the queue is rewritten by the next chunk
    }
}

// Pass 3 with 16-bit results, lane-major: lane l owns rows 8l .. 8l + 7 of the
// warp's chunk (one 16-byte load of results and one byte of the row bitmap,
// loaded a chunk ahead), so one warp scan of the lanes' pair counts gives every
// row its place, where the row-major form above scans once per round of 32 rows
// that holds a point in several polygons.  The chunk's pairs are put together in
// shared memory and written out as whole lines (lanes' own stretches are 64
// bytes apart).  Points in several polygons are queued, across chunks, and taken
// in full rounds of 32: their polygons come from the words that pass 1b packed,
// or the warp walks their lists (a wait per row of a lane, then one per chunk, was
// most of this kernel).  A chunk of more than kEmitStage pairs is written straight
// to its place.  500M points x 256 queries (17 % of the points in one or more):
// 2.77 ms row-major, 1.19 with a wait per chunk, 1.09 now; 100M x 1024 disks 257
// -> 154 us; 20M x 256 buffered queries 232 -> 65 us; 100M x 2000 cells (a
// pair per point) 204 -> 162 us for 1.0 GB, where a plain fill of its 0.8 GB
// takes 105.
//
// With SELF (small tables, a warp per chunk) chunk_off holds the chunks' totals,
// not their offsets: every CTA sums the totals before its first chunk itself
// (at most 8 B x kSmallChunks from L2), which saves the scan's launch.
// Pairs of the stage; a full chunk's lie nine apart per lane of eight (no bank
// conflict).  Disks, whose output is sparse, have a small one.
template <int KIND>
constexpr uint32_t kEmitStage = KIND == kDisk ? 96 : 320;
constexpr uint32_t kEmitQueue = kWChunk + 32; // a chunk's rows and a partial round
template <int KIND>
constexpr size_t kEmit16Warp = (kEmitStage<KIND> * 8 + size_t(kEmitQueue) * 12 + kWaveWords * 4 + 15) & ~size_t(15);
template <int KIND>
constexpr size_t kEmit16Smem = kWarps * kEmit16Warp<KIND>; // 49 KB (disks 35): four CTAs per SM
static_assert(kWItems == 8, "a lane's rows: one 16-byte load of 2-byte results");

template <bool FP32, bool SELF, int KIND>
__global__ void __launch_bounds__(kThreads, KIND == kNear ? 3 : 4) k_wemit16(const __grid_constant__ JoinLaunch a,
                                                         const unsigned long long *chunk_off, uint32_t nchunks,
                                                         const uint32_t *pend)
{
    __shared__ unsigned long long s_before[SELF ? kWarps : 1];
    extern __shared__ __align__(16) unsigned char s_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint2 *s_st = reinterpret_cast<uint2 *>(s_raw + warp * kEmit16Warp<KIND>);
    unsigned long long *s_o = reinterpret_cast<unsigned long long *>(s_st + kEmitStage<KIND>); // offset | count << 48
    uint32_t *s_q = reinterpret_cast<uint32_t *>(s_o + kEmitQueue); // rows of the table
    uint32_t *s_par = s_q + kEmitQueue;
    const uint64_t keep = policy_evict_last();
    const uint32_t nw = gridDim.x * kWarps, r0 = 8u * (uint32_t)lane;
    const unsigned short *res = reinterpret_cast<const unsigned short *>(a.res);
    const uint8_t *bits = reinterpret_cast<const uint8_t *>(pend);
    unsigned long long before = 0; // SELF: the pairs before this warp's chunk
    if (SELF) {
        const uint32_t c0 = blockIdx.x * kWarps;
        for (uint32_t i = threadIdx.x; i < c0; i += kThreads)
            before += chunk_off[i];
        before = warp_sum64(before);
        if (lane == 0)
            s_before[warp] = before;
        __syncthreads();
        before = 0;
        for (int w = 0; w < kWarps; ++w)
            before += s_before[w];
        for (int w = 0; w < warp && c0 + w < nchunks; ++w)
            before += chunk_off[c0 + w];
        if (c0 + warp == nchunks - 1 && lane == 0 && a.total)
            *a.total = before + chunk_off[nchunks - 1];
    }
    uint32_t nr[4], nm = 0; // the next chunk's results (two per word) and bitmap byte
    unsigned long long noff = 0;
    auto fetch = [&](uint32_t ch) {
        const uint64_t base = (uint64_t)ch * kWChunk;
        const uint32_t npts = ch < nchunks ? (uint32_t)min((uint64_t)kWChunk, a.n - base) : 0u;
        if (r0 + 8 <= npts) {
            const uint4 u = __ldcs(reinterpret_cast<const uint4 *>(res + base + r0));
            nr[0] = u.x, nr[1] = u.y, nr[2] = u.z, nr[3] = u.w;
        } else { // the table's ragged end
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t lo = r0 + 2 * k < npts ? __ldcs(res + base + r0 + 2 * k) : kRes16None;
                const uint32_t hi = r0 + 2 * k + 1 < npts ? __ldcs(res + base + r0 + 2 * k + 1) : kRes16None;
                nr[k] = lo | hi << 16;
            }
        }
        nm = ch < nchunks ? __ldcs(bits + (uint64_t)ch * 32 + lane) : 0u;
        if (!SELF)
            noff = ch < nchunks ? chunk_off[ch] : 0ull;
    };
    // writes the pairs of queued points [k0, k0 + m), m <= 32, one per lane
    auto several = [&](uint32_t k0, uint32_t m_) {
        const bool has = (uint32_t)lane < m_;
        const uint32_t row = s_q[k0 + (has ? lane : 0)], pid = a.pid0 + row;
        const unsigned long long oc = s_o[k0 + (has ? lane : 0)];
        unsigned long long o = oc & ((1ull << 48) - 1);
        const uint32_t c = uint32_t(oc >> 48);
        const bool packed = a.aux && c * a.aux_bits <= 64;
        if (has && packed) {
            unsigned long long ids = __ldcs(reinterpret_cast<const unsigned long long *>(a.aux) + row);
            for (uint32_t t = 0; t < c; ++t, ++o, ids >>= a.aux_bits)
                if (o < a.cap)
                    __stcs(a.pairs + o, make_uint2(pid, uint32_t(ids) & ((1u << a.aux_bits) - 1u)));
        }
        const bool walk = has && !packed; // the whole warp walks these points' lists together
        if (__any_sync(kFull, walk)) {
            const int2 p = walk ? a.pts[row] : make_int2(0, 0);
            const uint32_t w = walk ? resolve<KIND, KIND == kDisk>(a.ix, (uint32_t)p.x, (uint32_t)p.y, keep) : 0u;
            uint32_t t = 0, e = 0;
            walk_list_wave<FP32, KIND>(a.ix, (w >> 30) >= kCellList, w & kPayloadMask, p.x, p.y, t, e, keep, s_par,
                                       [&](uint32_t q) {
                                           if (o < a.cap)
                                               __stcs(a.pairs + o, make_uint2(pid, q));
                                           ++o;
                                       }, &a.near);
        }
        __syncwarp();
    };
    uint32_t qn = 0; // queued points, < 32 between chunks
    const unsigned long long pb = a.pair_base ? *a.pair_base : 0ull;
    fetch(blockIdx.x * kWarps + warp);
    for (uint32_t ch = blockIdx.x * kWarps + warp; ch < nchunks; ch += nw) {
        const uint64_t base = (uint64_t)ch * kWChunk;
        const uint32_t m = nm, pid0 = a.pid0 + (uint32_t)base + r0;
        const unsigned long long run = SELF ? before : noff + pb;
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            w[k] = nr[k];
        if (!SELF)
            fetch(ch + nw);
        // row k's result, and whether it is none (0xffff)
        auto r = [&](int k) { return k & 1 ? w[k >> 1] >> 16 : w[k >> 1] & 0xffffu; };
        auto none = [&](int k) { return (k & 1 ? w[k >> 1] : w[k >> 1] << 16) >= 0xffff0000u; };
        const bool any_m = __any_sync(kFull, m != 0);
        uint32_t mine = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            mine += none(k) ? 0u : 1u;
        if (any_m) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if ((m >> k) & 1u) // the count of a row in several polygons (never 0xffff: P is below it)
                    mine += r(k) - 1u;
        }
        if (kEmitStage<KIND> >= 9 * 32 && !any_m && __all_sync(kFull, mine == 8)) { // every row in one polygon
            uint2 *d = s_st + 9 * lane;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                d[k] = make_uint2(pid0 + k, r(k));
            __syncwarp();
            const uint2 *src = s_st + lane + (lane >> 3);
            if (run + kWChunk <= a.cap) {
                uint2 *out = a.pairs + run + lane;
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    __stcs(out + 32 * k, src[36 * k]);
            } else {
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (run + 32 * k + lane < a.cap)
                        __stcs(a.pairs + run + 32 * k + lane, src[36 * k]);
            }
            __syncwarp(); // the stage is rewritten by the next chunk
            continue;
        }
        uint32_t inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(kFull, inc, o);
            if (lane >= o)
                inc += v;
        }
        const uint32_t tot = __shfl_sync(kFull, inc, 31);
        if (tot == 0)
            continue;
        uint32_t at = inc - mine;
        const bool staged = tot <= kEmitStage<KIND>;
        if (!any_m && staged) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (!none(k))
                    s_st[at++] = make_uint2(pid0 + k, r(k));
        } else {
            uint32_t slot = __popc(m); // rows in several polygons: their places in the queue
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(kFull, slot, o);
                if (lane >= o)
                    slot += v;
            }
            const uint32_t nq = __shfl_sync(kFull, slot, 31);
            slot += qn - __popc(m);
            qn += nq;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if ((m >> k) & 1u) {
                    s_q[slot] = (uint32_t)base + r0 + k;
                    s_o[slot++] = (run + at) | (unsigned long long)r(k) << 48;
                    at += r(k);
                } else if (!none(k)) {
                    if (staged)
                        s_st[at] = make_uint2(pid0 + k, r(k));
                    else if (run + at < a.cap)
                        __stcs(a.pairs + run + at, make_uint2(pid0 + k, r(k)));
                    ++at;
                }
            }
        }
        __syncwarp();
        if (staged) {
            // whole lines; the places of queued points are written with what the
            // stage held, and with their pairs when their round comes
            const uint32_t n_out = run >= a.cap ? 0u : (uint32_t)min((unsigned long long)tot, a.cap - run);
            for (uint32_t i = lane; i < n_out; i += 32)
                __stcs(a.pairs + run + i, s_st[i]);
            __syncwarp();
        }
        if (qn >= 32) {
            uint32_t k0 = 0;
            for (; qn - k0 >= 32; k0 += 32)
                several(k0, 32);
            const uint32_t rem = qn - k0; // move the partial round (< 32, from k0 >= 32) to the front
            const uint32_t q = (uint32_t)lane < rem ? s_q[k0 + lane] : 0u;
            const unsigned long long oo = (uint32_t)lane < rem ? s_o[k0 + lane] : 0ull;
            __syncwarp();
            if ((uint32_t)lane < rem) {
                s_q[lane] = q;
                s_o[lane] = oo;
            }
            qn = rem;
            __syncwarp();
        }
    }
    if (qn)
        several(0, qn);
}

// ------------------------------------------------------ multi-request batches
// Serving answers several requests, each with its own index, in one pass over
// the points: the point table is read once per pass for the whole batch
// instead of once per request (the one-pass batched selection of §5.2,
// applied across requests).  Two passes, as in the Map of §5.1: the count pass
// counts every request's pairs per warp chunk (and the join requests'
// per-polygon counts); the per-request chunk totals are scanned; the emit pass
// resolves again and writes every request's pairs in (point, polygon) order
// from its chunk's offset.  As in k_warp, every warp works alone on its
// chunks (loaded once for all requests) and walks list points from a
// per-warp queue; the output never depends on the schedule.
constexpr uint32_t kMPending = 0xffffffffu; // a list point whose walk is queued
#ifndef SPX_MULTI_ITEMS
#define SPX_MULTI_ITEMS 4
#endif
constexpr int kMItems = SPX_MULTI_ITEMS;                      // points per lane per chunk
constexpr int kMChunk = 32 * kMItems;                         // consecutive points per warp chunk
// queues and offsets, then the words of walk_list_wave, per warp
constexpr size_t kMultiSmem =
    size_t(kWarps) * (kMChunk * (sizeof(uint4) + sizeof(unsigned long long)) + kWaveWords * sizeof(uint32_t));

// Does the cover bitmap let (px, py) reach a non-empty coarse cell?  False for
// points outside the box.
__device__ __forceinline__ bool covered(const IndexView &ix, int px, int py)
{
    if ((unsigned)px >= kBox || (unsigned)py >= kBox)
        return false;
    const uint32_t b = (((uint32_t)py >> ix.scv) << ix.cg) | ((uint32_t)px >> ix.scv);
    return (__ldg(ix.cover + (b >> 5)) >> (b & 31)) & 1u;
}

template <bool FP32, bool EMIT>
__global__ void __launch_bounds__(kThreads, 3) k_multi(const __grid_constant__ MultiLaunch m,
                                                    unsigned long long *chunk_tot, uint32_t nchunks, int use_hist)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint4 *s_q = reinterpret_cast<uint4 *>(s_raw) + warp * kMChunk; // (x, y, first entry) -> (count, first)
    unsigned long long *s_o = // emit pass: output offsets of queued points
        reinterpret_cast<unsigned long long *>(s_raw + size_t(kWarps) * kMChunk * sizeof(uint4)) + warp * kMChunk;
    uint32_t *s_par = reinterpret_cast<uint32_t *>(
                          s_raw + size_t(kWarps) * kMChunk * (sizeof(uint4) + sizeof(unsigned long long))) +
                      warp * kWaveWords;
    uint32_t *s_hist = reinterpret_cast<uint32_t *>(s_raw + kMultiSmem); // count pass: qbase[K] counters
    const uint64_t keep = policy_evict_last();
    const int K = m.K;
    uint32_t tests = 0, esc = 0, scanned = 0, emitted = 0;
    if (!EMIT && use_hist)
        for (uint32_t i = threadIdx.x; i < m.qbase[K]; i += kThreads)
            s_hist[i] = 0;
    __syncthreads();
    const uint32_t nw = gridDim.x * kWarps;
    for (uint32_t ch = blockIdx.x * kWarps + warp; ch < nchunks; ch += nw) {
        const uint64_t base = (uint64_t)ch * kMChunk;
        const uint32_t npts = (uint32_t)min((uint64_t)kMChunk, m.n - base);
        int2 p[kMItems];
#pragma unroll
        for (int j = 0; j < kMItems; ++j) {
            const uint32_t loc = j * 32 + lane;
            p[j] = loc < npts ? __ldcs(m.pts + base + loc) : make_int2(-1, -1);
            if (!EMIT)
                scanned += loc < npts ? (uint32_t)K : 0u;
        }
        for (int r = 0; r < K; ++r) {
            const IndexView &ix = m.ix[r];
            uint32_t c[kMItems], f[kMItems];
#pragma unroll
            for (int j = 0; j < kMItems; ++j) {
                const bool ok = covered(ix, p[j].x, p[j].y);
                const uint32_t cw = coarse_word(ix, ok ? (uint32_t)p[j].x : 0u, ok ? (uint32_t)p[j].y : 0u, keep);
                f[j] = ok ? cw : 0u;
            }
#pragma unroll
            for (int j = 0; j < kMItems; ++j) {
                const bool sub = (f[j] >> 30) == kCellSub;
                const uint32_t fw = fine_word(ix, sub ? f[j] : 0u, sub ? (uint32_t)p[j].x : 0u,
                                              sub ? (uint32_t)p[j].y : 0u, keep);
                f[j] = sub ? fw : f[j];
            }
            // one INSIDE polygon: done; a list: queued
            uint32_t qn = 0;
#pragma unroll
            for (int j = 0; j < kMItems; ++j) {
                const uint32_t kind = f[j] >> 30;
                const bool lst = kind == kCellList;
                c[j] = kind == kCellInsideOne ? 1u : 0u;
                const uint32_t bl = __ballot_sync(kFull, lst);
                if (lst) {
                    const uint32_t slot = qn + __popc(bl & lanemask_lt());
                    s_q[slot] = make_uint4((uint32_t)p[j].x, (uint32_t)p[j].y, f[j] & kPayloadMask, 0u);
                    c[j] = kMPending;
                    f[j] = slot;
                } else {
                    f[j] &= kPayloadMask;
                }
                qn += __popc(bl);
            }
            __syncwarp();
            unsigned long long *cnt = m.counts[r];
            uint32_t *h = s_hist + m.qbase[r];
            for (uint32_t k0 = 0; k0 < qn; k0 += 32) {
                const bool has = k0 + lane < qn;
                const uint4 it = s_q[has ? k0 + lane : k0]; // idle lanes walk nothing
                // the warp walks its lanes' lists together; the count pass counts a
                // point's further polygons here, its first one with the warp below
                uint32_t fq = 0, cq = 0, t_l = 0, e_l = 0;
                walk_list_wave<FP32>(ix, has, it.z, (int)it.x, (int)it.y, t_l, e_l, keep, s_par, [&](uint32_t q) {
                    if (cq == 0)
                        fq = q;
                    else if (!EMIT && cnt)
                        use_hist ? (void)atomicAdd(h + q, 1u) : (void)atomicAdd(cnt + q, 1ull);
                    ++cq;
                });
                if (!EMIT) {
                    tests += t_l;
                    esc += e_l;
                }
                __syncwarp();
                if (has)
                    s_q[k0 + lane] = make_uint4(cq, fq, 0u, 0u);
                __syncwarp();
            }
#pragma unroll
            for (int j = 0; j < kMItems; ++j)
                if (c[j] == kMPending) {
                    const uint4 q = s_q[f[j]];
                    c[j] = q.x;
                    f[j] = q.y;
                }
            __syncwarp(); // s_q is rewritten for the next request
            if (!EMIT) {
                uint32_t total = 0;
#pragma unroll
                for (int j = 0; j < kMItems; ++j) {
                    total += c[j];
                    if (!cnt)
                        continue;
                    // the first polygon of every point in any (further ones were counted by the walk)
                    if (!use_hist) // served tables are in row order: lanes rarely share a counter
                        global_add_warp(cnt, c[j] >= 1, f[j]);
                    else if (c[j] >= 1)
                        atomicAdd(h + f[j], 1u);
                }
                total = warp_sum32(total);
                if (lane == 0)
                    chunk_tot[(uint64_t)r * nchunks + ch] = total;
                continue;
            }
            // emit: pairs of request r in point order from the chunk's offset;
            // points in several polygons are queued and walked 32 at a time
            uint2 *out = m.pairs[r];
            const uint64_t cap = m.cap[r];
            unsigned long long run = chunk_tot[(uint64_t)r * nchunks + ch];
            uint32_t mq = 0;
#pragma unroll
            for (int j = 0; j < kMItems; ++j) {
                const uint32_t loc = j * 32 + lane, cj = c[j];
                uint32_t inc = cj;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t v = __shfl_up_sync(kFull, inc, o);
                    if (lane >= o)
                        inc += v;
                }
                const uint32_t wtot = __shfl_sync(kFull, inc, 31);
                const unsigned long long o = run + inc - cj;
                const uint32_t pid = (uint32_t)(base + loc);
                if (cj == 1 && o < cap)
                    out[o] = make_uint2(pid, f[j]);
                const uint32_t bl = __ballot_sync(kFull, cj > 1);
                if (cj > 1) {
                    const uint32_t slot = mq + __popc(bl & lanemask_lt());
                    s_q[slot] = make_uint4((uint32_t)p[j].x, (uint32_t)p[j].y, pid, 0u);
                    s_o[slot] = o;
                }
                mq += __popc(bl);
                emitted += cj;
                run += wtot;
            }
            __syncwarp();
            for (uint32_t k0 = 0; k0 < mq; k0 += 32) {
                // the whole warp walks the queued points' lists together
                const bool has = k0 + lane < mq;
                const uint4 it = has ? s_q[k0 + lane] : make_uint4(0u, 0u, 0u, 0u);
                unsigned long long o = has ? s_o[k0 + lane] : 0ull;
                const uint32_t w = has ? resolve(ix, it.x, it.y, keep) : 0u;
                uint32_t t_l = 0, e_l = 0;
                walk_list_wave<FP32>(ix, (w >> 30) == kCellList, w & kPayloadMask, (int)it.x, (int)it.y, t_l, e_l, keep,
                                     s_par, [&](uint32_t q) {
                                         if (o < cap)
                                             out[o] = make_uint2(it.z, q);
                                         ++o;
                                     });
            }
            __syncwarp(); // s_q is rewritten for the next request
        }
    }
    if (!EMIT && use_hist) {
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < m.qbase[K]; i += kThreads) {
            const uint32_t v = s_hist[i];
            if (!v)
                continue;
            int r = 0;
            while (r + 1 < K && i >= m.qbase[r + 1])
                ++r;
            atomicAdd(m.counts[r] + (i - m.qbase[r]), (unsigned long long)v);
        }
    }
    add_stats(m.stats, scanned, tests, esc, emitted);
}

// ------------------------------------------------------ batched selection
// Selection of points by many query polygons at once (§5.2 "Spatial
// Selection", one pass over the points for all queries).  The join runs once
// and yields (point, query) pairs in point order; the pairs are then
// partitioned by query, keeping point order: each super-tile (super_tile(cap)
// pairs) counts its pairs per query into a query-major table; an exclusive scan
// of the table in query-major order makes entry (q, s) the output position of
// super-tile s's first pair of query q; the emit kernel writes the point ids.
// Pairs per super-tile: 32768 while the output is large (the table then costs
// 8 B per 32768 / P pairs), halved while that leaves the chip without two
// tiles per SM, down to 1024: both kernels are chains of dependent steps per
// tile, and a small output was one or two of them (3M points x 16 queries,
// room for 207k ids: count + emit 170 -> 11.6 us; 84M ids of 256 queries keep
// 32768).
constexpr int kSuperTileMax = 32768, kSuperTileMin = 1024;
constexpr uint32_t kSuperTiles = 2 * 152;  // two per SM
constexpr int kSelMaxQ = 1024;            // queries per index (shared-memory counters)
constexpr int kPartTile = 4096;           // pairs that k_part_emit orders in shared memory at a time
constexpr int kPartRounds = kPartTile / kThreads; // rounds of 32 pairs per warp and tile
static_assert(kSelMaxQ == 4 * kThreads, "k_part_emit: at most four queries per thread");

uint32_t super_tile(uint64_t cap)
{
    uint32_t t = kSuperTileMax;
    while (t > kSuperTileMin && (cap + t - 1) / t < kSuperTiles)
        t >>= 1;
    return t;
}

__global__ void __launch_bounds__(kThreads) k_part_count(const uint2 *__restrict__ pairs,
                                                         const unsigned long long *total, uint64_t cap, uint32_t P,
                                                         unsigned long long *table, uint32_t n_super, uint32_t tile)
{
    extern __shared__ uint32_t s_cnt[]; // P counters
    for (uint32_t q = threadIdx.x; q < P; q += kThreads)
        s_cnt[q] = 0;
    __syncthreads();
    const unsigned long long n = min(*total, (unsigned long long)cap); // pairs past cap were not written
    const uint64_t base = (uint64_t)blockIdx.x * tile;
    const uint32_t m = base < n ? (uint32_t)min((unsigned long long)tile, n - base) : 0u;
    for (uint32_t j = threadIdx.x; j < ((m + 31) & ~31u); j += kThreads) { // whole warps take part
        const bool has = j < m;
        const uint32_t q = has ? __ldcg(&pairs[base + j].y) : 0u;
        hist_add_warp(s_cnt, has, q);
    }
    __syncthreads();
    for (uint32_t q = threadIdx.x; q < P; q += kThreads)
        table[(uint64_t)q * n_super + blockIdx.x] = s_cnt[q];
}

// Writes the ids of a super-tile's pairs at their queries' positions.  Pairs
// arrive in point order and neighbours rarely share a query, so writing each
// id straight to its list touches another sector per lane (84M ids: 2.04 ms,
// a quarter of the L2's sector rate and nothing else busy).  Instead the block
// orders kPartTile pairs by query in shared memory (stable: every warp ranks
// its own contiguous range with one match per round, a block scan turns
// the (query, warp) counts into places), then writes them in that order, so
// that consecutive threads write consecutive ids of a list (runs of 16 at 256
// queries).  Shared memory: kPartSmem(P).
constexpr size_t part_smem(uint32_t P)
{
    return size_t(P) * (8 + 8 + 2 * kWarps) + size_t(kPartTile) * (4 + 2);
}

__global__ void __launch_bounds__(kThreads, 4) k_part_emit(const uint2 *__restrict__ pairs,
                                                        const unsigned long long *total, uint32_t P,
                                                        const unsigned long long *table, uint32_t n_super,
                                                        uint32_t *ids, uint64_t cap, uint32_t tile)
{
    extern __shared__ __align__(16) unsigned char s_raw[];
    unsigned long long *s_run = reinterpret_cast<unsigned long long *>(s_raw); // P: next output position
    unsigned long long *s_off = s_run + P;                                    // P: position - place in the tile
    uint32_t *s_id = reinterpret_cast<uint32_t *>(s_off + P);                 // kPartTile ids in query order
    uint16_t *s_qy = reinterpret_cast<uint16_t *>(s_id + kPartTile);          // and their queries
    uint16_t *s_wc = s_qy + kPartTile;                                        // kWarps x P counts, then places
    __shared__ uint32_t s_wsum[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, bits = 32 - __clz(P - 1); // of a query (P = 1: none)
    const int kq = (P + kThreads - 1) / kThreads;
    const unsigned long long n = min(*total, (unsigned long long)cap); // pairs past cap were not written
    const uint64_t base = (uint64_t)blockIdx.x * tile;
    if (base >= n)
        return;
    const uint32_t mt = (uint32_t)min((unsigned long long)tile, n - base);
    for (uint32_t q = threadIdx.x; q < P; q += kThreads)
        s_run[q] = table[(uint64_t)q * n_super + blockIdx.x];
    for (uint32_t t0 = 0; t0 < mt; t0 += kPartTile) {
        const uint32_t m = min(mt - t0, (uint32_t)kPartTile);
        for (uint32_t i = threadIdx.x; i < kWarps * P / 2; i += kThreads)
            reinterpret_cast<uint32_t *>(s_wc)[i] = 0u; // kWarps is even
        __syncthreads();
        // 1. every warp counts its range per query and ranks its pairs
        const uint32_t span = (m + kThreads - 1) / kThreads * 32, w0 = warp * span, w1 = min(m, w0 + span);
        uint2 pr[kPartRounds]; // (id, query), the query's word then with the rank in its upper half
#pragma unroll
        for (int r = 0; r < kPartRounds; ++r) {
            const uint32_t j = w0 + r * 32 + lane;
            pr[r] = j < w1 ? __ldcs(&pairs[base + t0 + j]) : make_uint2(0u, 0xffffffffu);
        }
        uint16_t *wc = s_wc + warp * P;
#pragma unroll
        for (int r = 0; r < kPartRounds; ++r) {
            if (r * 32 >= span)
                break;
            const bool has = w0 + r * 32 + lane < w1;
            // the lanes of the same query, from a vote per bit of it (a match per
            // round, and 64 threads summing the warps' counts of 256 queries, took 827 us
            // of 84M ids, this 610)
            const uint32_t q = pr[r].y;
            uint32_t peers = __ballot_sync(kFull, has);
            for (int b = 0; b < bits; ++b) {
                const uint32_t v = __ballot_sync(kFull, (q >> b) & 1u);
                peers &= (q >> b) & 1u ? v : ~v;
            }
            const uint32_t before = has ? wc[q] : 0u;
            __syncwarp();
            if (has && lane == __ffs(peers) - 1)
                wc[q] = (uint16_t)(before + __popc(peers));
            __syncwarp();
            pr[r].y = q | (before + __popc(peers & lanemask_lt())) << 16;
        }
        __syncthreads();
        // 2. places: queries in order, within a query the warps in order
        uint32_t c4[4], mine = 0; // kq queries per thread
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t q = threadIdx.x * kq + k;
            c4[k] = 0;
            if (k < kq && q < P)
                for (int w = 0; w < kWarps; ++w)
                    c4[k] += s_wc[w * P + q];
            mine += c4[k];
        }
        uint32_t inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(kFull, inc, o);
            if (lane >= o)
                inc += v;
        }
        if (lane == 31)
            s_wsum[warp] = inc;
        __syncthreads();
        uint32_t at = inc - mine;
        for (int w = 0; w < warp; ++w)
            at += s_wsum[w];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t q = threadIdx.x * kq + k;
            if (k < kq && q < P) {
                s_off[q] = s_run[q] - at; // modulo 2^64: a place of the query is at or above `at`
                s_run[q] += c4[k];
                for (int w = 0; w < kWarps; ++w) {
                    const uint16_t c = s_wc[w * P + q];
                    s_wc[w * P + q] = (uint16_t)at;
                    at += c;
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kPartRounds; ++r)
            if (w0 + r * 32 + lane < w1) {
                const uint32_t q = pr[r].y & 0xffffu, pl = wc[q] + (pr[r].y >> 16);
                s_id[pl] = pr[r].x;
                s_qy[pl] = (uint16_t)q;
            }
        __syncthreads();
        // 3. out, in list order
        for (uint32_t i = threadIdx.x; i < m; i += kThreads) {
            const unsigned long long o = s_off[s_qy[i]] + i;
            if (o < cap)
                ids[o] = s_id[i];
        }
        __syncthreads(); // s_off and the places are rewritten by the next tile
    }
}

// offsets[q] = first position of query q (table entry (q, 0)), offsets[P] = total
__global__ void k_sel_offsets(const unsigned long long *table, uint32_t n_super, uint32_t P,
                              const unsigned long long *total, unsigned long long *offsets)
{
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q <= P; q += gridDim.x * blockDim.x)
        offsets[q] = q < P ? table[(uint64_t)q * n_super] : *total;
}

__global__ void __launch_bounds__(kPlainThreads) k_plain_write(JoinLaunch a, const unsigned long long *block_off)
{
    __shared__ uint32_t s_w[(kPlainThreads / 32)];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t idx = (uint64_t)blockIdx.x * kPlainThreads + threadIdx.x;
    uint32_t c = 0, first = 0, t = 0, e = 0;
    int2 p = make_int2(0, 0);
    const uint64_t keep = policy_evict_last();
    if (idx < a.n) {
        p = a.pts[idx];
        c = point_count<false>(a.ix, p.x, p.y, first, t, e, keep);
    }
    uint32_t inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(kFull, inc, o);
        if (lane >= o)
            inc += v;
    }
    if (lane == 31)
        s_w[warp] = inc;
    __syncthreads();
    uint32_t wpre = 0;
    for (int w = 0; w < warp; ++w)
        wpre += s_w[w];
    unsigned long long o = block_off[blockIdx.x] + wpre + inc - c;
    if (c == 1) {
        if (o < a.cap)
            a.pairs[o] = make_uint2((uint32_t)idx, first);
        if (a.counts)
            atomicAdd(a.counts + first, 1ull);
    } else if (c > 1) {
        point_emit<false>(a.ix, p.x, p.y, keep, [&](uint32_t q) {
            if (o < a.cap)
                a.pairs[o] = make_uint2((uint32_t)idx, q);
            ++o;
            if (a.counts)
                atomicAdd(a.counts + q, 1ull);
        });
    }
}

template <bool FP32, bool CLUSTERED>
cudaError_t launch_warp_kernel(const JoinLaunch &a, int use_hist, cudaStream_t s)
{
    static bool done[64] = {};
    const uint64_t nchunks = (a.n + kWChunk - 1) / kWChunk;
    if (nchunks >= (1ull << 32))
        return cudaErrorInvalidValue;
    const size_t smem = kWarpSmem + (use_hist ? sizeof(uint32_t) * a.ix.P : 0);
    auto kern = k_warp<FP32, CLUSTERED>;
    cudaError_t e = smem_opt_in(kern, kWarpSmem + sizeof(uint32_t) * kHistMax, done);
    if (e != cudaSuccess)
        return e;
    const uint32_t nblk = uint32_t((nchunks + kWarps - 1) / kWarps);
    kern<<<persistent_grid(kern, kThreads, smem, nblk), kThreads, smem, s>>>(a, uint32_t(nchunks), use_hist);
    return cudaGetLastError();
}

// The directory stage of the count aggregate over a cell-clustered table (2^c
// grid, c >= g).  A cell inside a coarse cell INSIDE one polygon adds its whole row
// range to that polygon (its points need not be read); an empty one adds nothing;
// one in a mixed coarse cell marks its rows in the bitmap, for k_walk<ALL>.  The
// points of the cells counted here, and of the bin outside the box, go into the
// scanned-points counter.  A warp takes strips of 32 columns and kDirRows rows, a
// lane per column, kDirCells rows at a time: going down its column a lane stays in
// one polygon for many rows and adds to that polygon's counter when it leaves it.
// (32 neighbouring cells of a row mostly hold two polygons, and an atomic per cell
// was two thirds of this stage: 2^26 cells and 40000 polygons, 656 -> 331 us; the
// marks are most of the rest.)
constexpr int kDirCells = 4;
constexpr uint32_t kDirRows = 64;
__global__ void __launch_bounds__(256) k_agg_cells(const unsigned long long *cell_end, int c, IndexView ix,
                                                   unsigned long long *counts, uint32_t *rows,
                                                   unsigned long long *stats)
{
    const uint32_t side = 1u << c, lane = threadIdx.x & 31;
    const uint32_t strips = (side + 31) / 32, bands = (side + kDirRows - 1) / kDirRows;
    const int sh = c - ix.gc;
    unsigned long long done_pts = 0;
    for (uint32_t u = blockIdx.x * 8 + (threadIdx.x >> 5); u < strips * bands; u += gridDim.x * 8) {
        const uint32_t x = (u % strips) * 32 + lane, y0 = (u / strips) * kDirRows, y1 = min(side, y0 + kDirRows);
        uint32_t cur_q = 0, cur_n = 0; // this lane's polygon and its points so far
        for (uint32_t yb = y0; yb < y1; yb += kDirCells) {
            uint32_t s0[kDirCells], s1[kDirCells], w[kDirCells]; // a cell's rows [s0, s1) and its coarse word
#pragma unroll
            for (int j = 0; j < kDirCells; ++j) {
                const uint32_t k = ((yb + j) << c) + x;
                const bool in = x < side && yb + j < y1;
                s1[j] = in ? (uint32_t)cell_end[k] : 0u;
                s0[j] = in && lane == 0 && k ? (uint32_t)cell_end[k - 1] : 0u;
            }
#pragma unroll
            for (int j = 0; j < kDirCells; ++j) {
                const uint32_t up = __shfl_up_sync(kFull, s1[j], 1);
                s0[j] = lane ? up : s0[j];
                w[j] = 0;
                if (s1[j] > s0[j])
                    w[j] = ix.cell[(((yb + j) >> sh) << ix.gc) | (x >> sh)];
            }
#pragma unroll
            for (int j = 0; j < kDirCells; ++j) {
                const uint32_t num = s1[j] > s0[j] ? s1[j] - s0[j] : 0u;
                const uint32_t kind = w[j] >> 30, q = w[j] & kPayloadMask;
                const bool sub = kind == kCellSub; // a cell without points has w = 0
                done_pts += sub ? 0u : num;
                if (kind == kCellInsideOne && in_bounds(q < ix.P, ix)) {
                    if (q != cur_q) {
                        if (cur_n)
                            atomicAdd(counts + cur_q, (unsigned long long)cur_n);
                        cur_q = q;
                        cur_n = 0;
                    }
                    cur_n += num;
                }
                if (!__any_sync(kFull, sub))
                    continue;
                // rows of a cell in a mixed coarse cell; ranges over two words by the warp
                const uint32_t r0 = s0[j], r1 = sub ? s1[j] - 1 : s0[j];
                auto mark = [&](uint32_t wd, uint32_t a, uint32_t z) {
                    const uint32_t lo = wd == (a >> 5) ? a & 31u : 0u, hi = wd == (z >> 5) ? z & 31u : 31u;
                    if (hi - lo == 31)
                        rows[wd] = 0xffffffffu; // no other cell's rows here
                    else
                        atomicOr(rows + wd, (0xffffffffu >> (31 - (hi - lo))) << lo);
                };
                const bool wide = (r1 >> 5) - (r0 >> 5) > 1;
                if (sub && !wide) {
                    mark(r0 >> 5, r0, r1);
                    if ((r1 >> 5) != (r0 >> 5))
                        mark(r1 >> 5, r0, r1);
                }
                for (uint32_t todo = __ballot_sync(kFull, sub && wide); todo; todo &= todo - 1) {
                    const int src = __ffs(todo) - 1;
                    const uint32_t a = __shfl_sync(kFull, r0, src), z = __shfl_sync(kFull, r1, src);
                    for (uint32_t wd = (a >> 5) + lane; wd <= (z >> 5); wd += 32)
                        mark(wd, a, z);
                }
            }
        }
        // the strip's last polygons: one atomic where the lanes share theirs
        const uint32_t m = __ballot_sync(kFull, cur_n != 0);
        if (m) {
            const uint32_t q0 = __shfl_sync(kFull, cur_q, __ffs(m) - 1);
            if (!__any_sync(kFull, cur_n && cur_q != q0)) {
                const uint32_t t = __reduce_add_sync(kFull, cur_n); // rows: below 2^32 in all
                if ((int)lane == __ffs(m) - 1)
                    atomicAdd(counts + q0, (unsigned long long)t);
            } else if (cur_n) {
                atomicAdd(counts + cur_q, (unsigned long long)cur_n);
            }
        }
    }
    // the bin of points outside the box: in no polygon
    if (blockIdx.x == 0 && threadIdx.x == 0)
        done_pts += cell_end[(size_t(1) << (2 * c))] - cell_end[(size_t(1) << (2 * c)) - 1];
    __shared__ unsigned long long s_done;
    if (threadIdx.x == 0)
        s_done = 0ull;
    __syncthreads();
    done_pts = warp_sum64(done_pts);
    if (lane == 0 && done_pts)
        atomicAdd(&s_done, done_pts);
    __syncthreads();
    if (threadIdx.x == 0 && s_done) {
        atomicAdd(stats + kStatPoints, s_done);
        atomicAdd(stats + kStatDirPoints, s_done);
    }
}

// Pass 1 of the join (1a resolve, 1b walk).  pend: 8 words per chunk (the
// bitmap of the rows pass 1b tests).  mid (or null): an event recorded between
// the two kernels.
template <bool FP32, int OUT, int KIND>
cudaError_t launch_pass1_as(const JoinLaunch &a, uint32_t *pend, cudaStream_t s, cudaEvent_t mid)
{
    static bool done_r[4][64] = {};
    const uint64_t nchunks = (a.n + kWChunk - 1) / kWChunk;
    if (a.n >= (1ull << 32))
        return cudaErrorInvalidValue; // rows are 32-bit
    const int use_hist = (a.counts != nullptr && a.ix.P <= (uint32_t)kHistMax) ? 1 : 0;
    const size_t hsm = use_hist ? sizeof(uint32_t) * a.ix.P : 0;
    cudaError_t e;
    if (reinterpret_cast<uintptr_t>(a.pts) & 15)
        return cudaErrorMisalignedAddress; // bulk copies of whole chunks start 16-byte aligned
    // the largest shared memory a CTA may take
    int dev = 0, smem_max = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    // head: this launch's shared memory before the counters; head_max: the
    // most any launch of the kernel takes (the opt-in, set once per device,
    // must cover every later call, whatever its index)
    auto launch = [&](auto kr, int threads, size_t head, size_t head_max, bool (&done)[64]) -> cudaError_t {
        const size_t smem = head + hsm;
        cudaError_t err =
            smem_opt_in(kr, std::min<size_t>(size_t(smem_max), head_max + sizeof(uint32_t) * kHistMax), done);
        if (err != cudaSuccess)
            return err;
        const uint32_t nblk = uint32_t((nchunks + threads / 32 - 1) / (threads / 32));
        kr<<<persistent_grid(kr, threads, smem, nblk), threads, smem, s>>>(a, pend, uint32_t(nchunks), use_hist);
        return cudaGetLastError();
    };
    constexpr int WS = kResolveSumThreads / 32;
    if (a.ix.use_sum) {
        // beside the summary, shared memory holds one chunk buffer per warp
        // at most, too shallow to hide a bulk copy: L2 prefetches instead
        e = launch(k_resolve_sum<OUT, KIND == kDisk>, kResolveSumThreads,
                   resolve_smem_head(WS, true, a.ix.sg, false), resolve_smem_head(WS, true, kSumLog2, false), done_r[2]);
    } else {
        const size_t head = kTmaPoints ? resolve_smem_head(kWarps, false, 0, true) : 0;
        e = launch(k_resolve<kThreads, kTmaPoints, OUT, KIND == kDisk>, kThreads, head, head, done_r[3]);
    }
    if (e != cudaSuccess) // pass 1b must not run on what an earlier call left in the scratch
        return e;
    if (mid)
        cudaEventRecord(mid, s);
    return launch_walk<FP32, OUT, KIND>(a, pend, s); // pass 1b
}

// Calls f(fp32, kind) with the launch's two switches as compile-time values
// (disk tests are in int64 alone).
template <class F>
cudaError_t with_switches(const JoinLaunch &a, F f)
{
    using std::integral_constant;
    if (a.near.disk)
        return f(std::true_type{}, integral_constant<int, kDisk>{});
    if (a.near.rad)
        return a.fp32 ? f(std::true_type{}, integral_constant<int, kNear>{}) : f(std::false_type{}, integral_constant<int, kNear>{});
    return a.fp32 ? f(std::true_type{}, integral_constant<int, kPoly>{}) : f(std::false_type{}, integral_constant<int, kPoly>{});
}

cudaError_t launch_pass1(const JoinLaunch &a, uint32_t *pend, cudaStream_t s, cudaEvent_t mid, bool count_only)
{
    return with_switches(a, [&](auto fp32, auto kind) -> cudaError_t {
        constexpr bool F = decltype(fp32)::value;
        constexpr int N = decltype(kind)::value;
        if constexpr (N == kDisk) {
            if (pend && a.ix.P <= kDiskSplit)
                return count_only ? launch_pass1_as<F, kOutCount, N>(a, pend, s, mid)
                                  : launch_pass1_as<F, kOut16, N>(a, pend, s, mid);
            const cudaError_t e = count_only ? launch_disk_pass1<kOutCount>(a, nullptr, s)
                                  : a.narrow ? launch_disk_pass1<kOut16>(a, pend, s)
                                             : launch_disk_pass1<kOut32>(a, pend, s);
            if (mid)
                cudaEventRecord(mid, s);
            return e;
        } else {
            return count_only ? launch_pass1_as<F, kOutCount, N>(a, pend, s, mid)
                   : a.narrow ? launch_pass1_as<F, kOut16, N>(a, pend, s, mid)
                              : launch_pass1_as<F, kOut32, N>(a, pend, s, mid);
        }
    });
}

// Exclusive scan of n values in place; the total goes to *total.  part: at
// least scan_partials(n) + 1 values of scratch.
uint64_t scan_partials(uint64_t n) { return (n + kScanChunk - 1) / kScanChunk; }

cudaError_t launch_scan(unsigned long long *v, uint64_t n, unsigned long long *total, unsigned long long *part,
                        cudaStream_t s)
{
    if (n <= 4 * kScanChunk) {
        k_scan<<<1, 1024, 0, s>>>(v, n, total);
        return cudaGetLastError();
    }
    const uint64_t nb = scan_partials(n);
    if (nb >= (1ull << 31))
        return cudaErrorInvalidValue;
    k_scan_partials<<<(unsigned)nb, 1024, 0, s>>>(v, n, part);
    k_scan<<<1, 1024, 0, s>>>(part, nb, total);
    k_scan_apply<<<(unsigned)nb, 1024, 0, s>>>(v, n, part);
    return cudaGetLastError();
}

} // namespace

// The bounded wait of pass 1a's bulk-copy staging on a barrier that nothing
// completes (no copy is issued): after `tries` polls it reports kErrTimeout.
__global__ void k_wait_check(unsigned *err, uint32_t tries)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0)
        mbar_init(&bar, 1);
    __syncwarp();
    if (!mbar_wait(&bar, 0, tries) && threadIdx.x == 0)
        atomicOr(err, kErrTimeout);
}

cudaError_t launch_wait_check(unsigned *err, uint32_t tries, cudaStream_t s)
{
    k_wait_check<<<1, 32, 0, s>>>(err, tries);
    return cudaGetLastError();
}

uint64_t scan_part_words(uint64_t n) { return scan_partials(n) + 2; }
cudaError_t launch_exclusive_scan(unsigned long long *v, uint64_t n, unsigned long long *total,
                                  unsigned long long *part, cudaStream_t s)
{
    return launch_scan(v, n, total, part, s);
}

// Deterministic sample for the tuner: dst[i] = src[i * stride], i < m.
__global__ void __launch_bounds__(256) k_gather_stride(const int2 *__restrict__ src, uint64_t stride,
                                                     int2 *__restrict__ dst, uint64_t m)
{
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < m; i += (uint64_t)gridDim.x * 256)
        dst[i] = src[i * stride];
}

cudaError_t launch_gather_stride(const int2 *src, uint64_t n, int2 *dst, uint64_t m, cudaStream_t s)
{
    if (m == 0)
        return cudaSuccess;
    if (m > n)
        return cudaErrorInvalidValue;
    const uint64_t stride = n / m; // (m - 1) * stride < n
    const uint64_t blocks = std::min<uint64_t>((m + 255) / 256, uint64_t(device_sm_count()) * 8);
    k_gather_stride<<<unsigned(blocks), 256, 0, s>>>(src, stride, dst, m);
    return cudaGetLastError();
}

// ------------------------------------------------------ disk index, built on the device
// The same arrays as the host build (build_disk_index): for every disk, every
// cell of its clipped bounding box is classified exactly in int64 (the cell's
// integer point nearest the centre beyond r: no entry; its farthest corner
// within r: INSIDE; else BOUNDARY); the (cell, disk) records are bucketed by
// cell; a cell with one INSIDE record gets a kind-1 word, any other non-empty
// cell a list (n, then the records in disk order), lists laid out in cell
// order after a reserved word 0.  No kernel here waits on another.
struct DiskBox {
    uint32_t i0, j0, w, h; // first cell column / row and the box's size in cells (w = 0: no cell)
};

__device__ __forceinline__ DiskBox disk_box(const int4 &d, int sh)
{
    const long long last = (long long)kBox - 1;
    const long long xlo = max(0ll, (long long)d.x - d.z), xhi = min(last, (long long)d.x + d.z);
    const long long ylo = max(0ll, (long long)d.y - d.z), yhi = min(last, (long long)d.y + d.z);
    if (xlo > xhi || ylo > yhi)
        return {0u, 0u, 0u, 0u};
    const uint32_t i0 = (uint32_t)(xlo >> sh), j0 = (uint32_t)(ylo >> sh);
    return {i0, j0, (uint32_t)(xhi >> sh) - i0 + 1, (uint32_t)(yhi >> sh) - j0 + 1};
}

// Does disk d reach cell (i, j) of side 2^sh, and does it hold the whole cell?
__device__ __forceinline__ bool disk_cell(const int4 &d, uint32_t i, uint32_t j, int sh, bool &inside)
{
    const long long S = 1ll << sh, x0 = (long long)i << sh, y0 = (long long)j << sh, x1 = x0 + S - 1,
                    y1 = y0 + S - 1;
    const long long cx = d.x, cy = d.y, rr = (long long)d.z * d.z;
    const long long nx = min(max(cx, x0), x1) - cx, ny = min(max(cy, y0), y1) - cy;
    if (nx * nx + ny * ny > rr)
        return false;
    const long long fx = max(cx - x0, x1 - cx), fy = max(cy - y0, y1 - cy);
    inside = fx * fx + fy * fy <= rr;
    return true;
}

// Records per disk (a block per disk, its threads over the box's cells) and
// the number of BOUNDARY records.
__global__ void __launch_bounds__(256) k_dbuild_count(const int4 *disk, uint32_t Q, int g,
                                                      unsigned long long *rec_cnt, unsigned long long *n_bnd)
{
    __shared__ unsigned long long s_c, s_b;
    const int sh = kBoxLog2 - g;
    for (uint32_t q = blockIdx.x; q < Q; q += gridDim.x) {
        if (threadIdx.x == 0)
            s_c = s_b = 0;
        __syncthreads();
        const int4 d = disk[q];
        const DiskBox b = disk_box(d, sh);
        const uint64_t n = (uint64_t)b.w * b.h;
        unsigned long long c = 0, bn = 0;
        for (uint64_t t = threadIdx.x; t < n; t += blockDim.x) {
            bool in = false;
            if (disk_cell(d, b.i0 + (uint32_t)(t % b.w), b.j0 + (uint32_t)(t / b.w), sh, in)) {
                ++c;
                bn += in ? 0u : 1u;
            }
        }
        c = warp_sum64(c);
        bn = warp_sum64(bn);
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&s_c, c);
            atomicAdd(&s_b, bn);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            rec_cnt[q] = s_c;
            if (s_b)
                atomicAdd(n_bnd, s_b);
        }
        __syncthreads();
    }
}

// Records (cell, disk << 1 | boundary) at each disk's offset; per-cell record
// counts and an OR of their boundary flags.
__global__ void __launch_bounds__(256) k_dbuild_write(const int4 *disk, uint32_t Q, int g,
                                                      const unsigned long long *rec_off, uint2 *rec,
                                                      uint32_t *cell_cnt, uint32_t *cell_bnd)
{
    __shared__ unsigned long long s_pos;
    const int sh = kBoxLog2 - g;
    for (uint32_t q = blockIdx.x; q < Q; q += gridDim.x) {
        if (threadIdx.x == 0)
            s_pos = 0;
        __syncthreads();
        const int4 d = disk[q];
        const DiskBox b = disk_box(d, sh);
        const uint64_t n = (uint64_t)b.w * b.h;
        const unsigned long long base = rec_off[q];
        for (uint64_t t = threadIdx.x; t < n; t += blockDim.x) {
            const uint32_t i = b.i0 + (uint32_t)(t % b.w), j = b.j0 + (uint32_t)(t / b.w);
            bool in = false;
            if (disk_cell(d, i, j, sh, in)) {
                const uint32_t c = (j << g) | i;
                rec[base + atomicAdd(&s_pos, 1ull)] = make_uint2(c, (q << 1) | (in ? 0u : 1u));
                atomicAdd(cell_cnt + c, 1u);
                if (!in)
                    atomicOr(cell_bnd + c, 1u);
            }
        }
        __syncthreads();
    }
}

// Words of the entry list of every cell that needs one (0 for the others).
__global__ void k_dbuild_words(uint32_t ncell, const uint32_t *cell_cnt, const uint32_t *cell_bnd,
                               unsigned long long *list_words)
{
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
        const uint32_t n = cell_cnt[c];
        list_words[c] = (n >= 2 || (n == 1 && cell_bnd[c])) ? n + 1ull : 0ull;
    }
}

// List cells: their word and list length (after the reserved word 0).
__global__ void k_dbuild_cells(uint32_t ncell, const uint32_t *cell_cnt, const uint32_t *cell_bnd,
                               const unsigned long long *list_off, uint32_t *cell_word, uint32_t *ent)
{
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
        const uint32_t n = cell_cnt[c];
        if (n >= 2 || (n == 1 && cell_bnd[c])) {
            const uint32_t off = 1u + (uint32_t)list_off[c];
            cell_word[c] = (kCellList << 30) | off;
            ent[off] = n;
        }
    }
}

// Every record to its cell: the word of a one-INSIDE cell, else the next slot
// of the cell's list (sorted afterwards).
__global__ void k_dbuild_scatter(uint64_t R, const uint2 *rec, const uint32_t *cell_cnt, const uint32_t *cell_bnd,
                                 const unsigned long long *list_off, uint32_t *cursor, uint32_t *cell_word,
                                 uint32_t *ent)
{
    for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < R; k += (uint64_t)gridDim.x * blockDim.x) {
        const uint2 r = rec[k];
        if (cell_cnt[r.x] == 1 && !cell_bnd[r.x])
            cell_word[r.x] = (kCellInsideOne << 30) | (r.y >> 1);
        else
            ent[2u + (uint32_t)list_off[r.x] + atomicAdd(cursor + r.x, 1u)] = r.y;
    }
}

// Each list in disk order (insertion sort: lists are short).
__global__ void k_dbuild_sort(uint32_t ncell, const uint32_t *cell_word, uint32_t *ent)
{
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
        const uint32_t w = cell_word[c];
        if ((w >> 30) != kCellList)
            continue;
        uint32_t *l = ent + (w & kPayloadMask) + 1;
        const uint32_t n = l[-1];
        for (uint32_t a = 1; a < n; ++a) {
            const uint32_t v = l[a];
            uint32_t b = a;
            for (; b > 0 && l[b - 1] > v; --b)
                l[b] = l[b - 1];
            l[b] = v;
        }
    }
}

// Cover bitmap: a bit per block of cells that holds a non-empty cell.
__global__ void k_dbuild_cover(uint32_t ncell, int g, int cg, const uint32_t *cell_word, uint32_t *cover)
{
    for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < ncell; c += gridDim.x * blockDim.x) {
        if (!cell_word[c])
            continue;
        const uint32_t cx = c & ((1u << g) - 1), cy = c >> g;
        const uint32_t b = ((cy >> (g - cg)) << cg) | (cx >> (g - cg));
        atomicOr(cover + (b >> 5), 1u << (b & 31));
    }
}

int build_disk_index_device(const int4 *disks_host, uint32_t Q, int g, DiskIndexDev &out, cudaError_t &cerr)
{
    out = DiskIndexDev{};
    cerr = cudaSuccess;
    const uint32_t ncell = 1u << (2 * g);
    const int cg = g < kCoverLog2 ? g : kCoverLog2;
    const size_t cover_words = ((size_t(1) << (2 * cg)) / 32) > 0 ? ((size_t(1) << (2 * cg)) / 32) : 1;
    const size_t nd = Q ? Q : 1;
    const uint64_t nparts = scan_partials(ncell > nd ? ncell : nd) + 2;
    // temporaries: disks | per-disk record counts | totals | scan partials |
    // per-cell counts, flags, cursors | per-cell list words
    auto up = [](size_t v) { return (v + 255) & ~size_t(255); };
    const size_t t_disk = up(nd * sizeof(int4)), t_cnt = up((nd + 1) * 8), t_tot = up(3 * 8), t_part = up(nparts * 8),
                 t_cell = up(size_t(ncell) * 4), t_words = up(size_t(ncell) * 8);
    char *tmp = nullptr, *recm = nullptr;
    auto done = [&](int status, cudaError_t e) {
        cerr = e;
        if (recm)
            cudaFree(recm);
        if (tmp)
            cudaFree(tmp);
        if (status && out.mem) {
            cudaFree(out.mem);
            out.mem = nullptr;
        }
        return status;
    };
    cudaError_t e = cudaMalloc(&tmp, t_disk + t_cnt + t_tot + t_part + 3 * t_cell + t_words);
    if (e != cudaSuccess)
        return done(2, e);
    int4 *d_disk = reinterpret_cast<int4 *>(tmp);
    auto *rec_cnt = reinterpret_cast<unsigned long long *>(tmp + t_disk);
    auto *tot = reinterpret_cast<unsigned long long *>(tmp + t_disk + t_cnt); // records, list words, boundary
    auto *part = reinterpret_cast<unsigned long long *>(tmp + t_disk + t_cnt + t_tot);
    auto *cell_cnt = reinterpret_cast<uint32_t *>(tmp + t_disk + t_cnt + t_tot + t_part);
    auto *cell_bnd = reinterpret_cast<uint32_t *>(tmp + t_disk + t_cnt + t_tot + t_part + t_cell);
    auto *cursor = reinterpret_cast<uint32_t *>(tmp + t_disk + t_cnt + t_tot + t_part + 2 * t_cell);
    auto *words = reinterpret_cast<unsigned long long *>(tmp + t_disk + t_cnt + t_tot + t_part + 3 * t_cell);
    if ((e = cudaMemcpy(d_disk, disks_host, nd * sizeof(int4), cudaMemcpyHostToDevice)) != cudaSuccess ||
        (e = cudaMemset(tot, 0, 3 * 8)) != cudaSuccess || (e = cudaMemset(cell_cnt, 0, 3 * t_cell)) != cudaSuccess)
        return done(2, e);
    const int sms = device_sm_count();
    const unsigned dblocks = Q ? (Q < unsigned(sms * 8) ? Q : unsigned(sms * 8)) : 1u;
    const unsigned cblocks = unsigned((ncell + 255) / 256 < uint32_t(sms * 16) ? (ncell + 255) / 256 : sms * 16);
    unsigned long long R = 0, T = 0, nb = 0;
    if (Q) {
        k_dbuild_count<<<dblocks, 256>>>(d_disk, Q, g, rec_cnt, tot + 2);
        if ((e = cudaGetLastError()) != cudaSuccess || (e = launch_scan(rec_cnt, Q, tot, part, 0)) != cudaSuccess ||
            (e = cudaMemcpy(&R, tot, 8, cudaMemcpyDeviceToHost)) != cudaSuccess)
            return done(2, e);
    }
    if (R) {
        if ((e = cudaMalloc(&recm, R * sizeof(uint2))) != cudaSuccess)
            return done(2, e);
        k_dbuild_write<<<dblocks, 256>>>(d_disk, Q, g, rec_cnt, reinterpret_cast<uint2 *>(recm), cell_cnt, cell_bnd);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return done(2, e);
    }
    k_dbuild_words<<<cblocks, 256>>>(ncell, cell_cnt, cell_bnd, words);
    if ((e = cudaGetLastError()) != cudaSuccess || (e = launch_scan(words, ncell, tot + 1, part, 0)) != cudaSuccess ||
        (e = cudaMemcpy(&T, tot + 1, 8, cudaMemcpyDeviceToHost)) != cudaSuccess ||
        (e = cudaMemcpy(&nb, tot + 2, 8, cudaMemcpyDeviceToHost)) != cudaSuccess)
        return done(2, e);
    const uint64_t E = 1 + T;
    if (E > kPayloadMask)
        return done(1, cudaSuccess);
    // the index's own allocation: cells | entries | disks | cover, as the host path lays it out
    const size_t b_cell = size_t(ncell) * 4, b_ent = size_t(E) * 4, b_disk = nd * sizeof(int4), b_cover = cover_words * 4;
    out.bytes = up(b_cell) + up(b_ent) + up(b_disk) + up(b_cover);
    if ((e = cudaMalloc(&out.mem, out.bytes)) != cudaSuccess) {
        out.mem = nullptr;
        return done(2, e);
    }
    char *m = static_cast<char *>(out.mem);
    out.cell = reinterpret_cast<uint32_t *>(m);
    out.ent = reinterpret_cast<uint32_t *>(m + up(b_cell));
    out.disk = reinterpret_cast<int4 *>(m + up(b_cell) + up(b_ent));
    out.cover = reinterpret_cast<uint32_t *>(m + up(b_cell) + up(b_ent) + up(b_disk));
    if ((e = cudaMemset(out.cell, 0, b_cell)) != cudaSuccess || (e = cudaMemset(out.ent, 0, b_ent)) != cudaSuccess ||
        (e = cudaMemset(out.cover, 0, b_cover)) != cudaSuccess ||
        (e = cudaMemcpy(out.disk, d_disk, b_disk, cudaMemcpyDeviceToDevice)) != cudaSuccess)
        return done(2, e);
    k_dbuild_cells<<<cblocks, 256>>>(ncell, cell_cnt, cell_bnd, words, out.cell, out.ent);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return done(2, e);
    if (R) {
        const unsigned rblocks = unsigned((R + 255) / 256 < uint64_t(sms * 16) ? (R + 255) / 256 : sms * 16);
        k_dbuild_scatter<<<rblocks, 256>>>(R, reinterpret_cast<const uint2 *>(recm), cell_cnt, cell_bnd, words, cursor,
                                           out.cell, out.ent);
        k_dbuild_sort<<<cblocks, 256>>>(ncell, out.cell, out.ent);
    }
    k_dbuild_cover<<<cblocks, 256>>>(ncell, g, cg, out.cell, out.cover);
    if ((e = cudaGetLastError()) != cudaSuccess || (e = cudaDeviceSynchronize()) != cudaSuccess)
        return done(2, e);
    out.n_ent = E;
    out.n_boundary = nb;
    out.n_inside = R - nb;
    return done(0, cudaSuccess);
}

// ------------------------------------------------------ clustered point table
// Counting sort of a point table by grid cell (row-major cells of a 2^c x 2^c
// grid; points outside the box go to one last bin).  Lanes of a warp with the
// same key share one atomic.
__device__ __forceinline__ uint32_t cell_key(int2 p, int c)
{
    if ((unsigned)p.x >= kBox || (unsigned)p.y >= kBox)
        return 1u << (2 * c);
    const int sh = kBoxLog2 - c;
    return (((uint32_t)p.y >> sh) << c) | ((uint32_t)p.x >> sh);
}

__global__ void __launch_bounds__(256) k_cell_hist(const int2 *__restrict__ pts, uint64_t n, int c,
                                                 unsigned long long *cnt)
{
    const uint64_t stride = (uint64_t)gridDim.x * 256;
    for (uint64_t i0 = (uint64_t)blockIdx.x * 256 + (threadIdx.x & ~31u); i0 < n; i0 += stride) {
        const uint64_t i = i0 + (threadIdx.x & 31);
        const bool has = i < n;
        const uint32_t key = has ? cell_key(__ldcs(pts + i), c) : 0xffffffffu;
        const uint32_t peers = __match_any_sync(kFull, key);
        if (has && (int)(threadIdx.x & 31) == __ffs(peers) - 1)
            atomicAdd(cnt + key, (unsigned long long)__popc(peers));
    }
}

__global__ void __launch_bounds__(256) k_cell_scatter(const int2 *__restrict__ pts, uint64_t n, int c,
                                                    unsigned long long *cursor, int2 *__restrict__ out)
{
    const uint64_t stride = (uint64_t)gridDim.x * 256;
    const int lane = threadIdx.x & 31;
    for (uint64_t i0 = (uint64_t)blockIdx.x * 256 + (threadIdx.x & ~31u); i0 < n; i0 += stride) {
        const uint64_t i = i0 + lane;
        const bool has = i < n;
        const int2 p = has ? __ldcs(pts + i) : make_int2(-1, -1);
        const uint32_t key = has ? cell_key(p, c) : 0xffffffffu;
        const uint32_t peers = __match_any_sync(kFull, key);
        const int leader = __ffs(peers) - 1;
        unsigned long long base = 0;
        if (has && lane == leader)
            base = atomicAdd(cursor + key, (unsigned long long)__popc(peers));
        base = __shfl_sync(kFull, base, leader);
        if (has)
            out[base + __popc(peers & lanemask_lt())] = p;
    }
}

size_t cluster_scratch_bytes(int c)
{
    const uint64_t bins = (uint64_t(1) << (2 * c)) + 1;
    return size_t(bins + scan_partials(bins) + 2) * 8 + 64;
}

cudaError_t launch_cluster(const int2 *pts, uint64_t n, int c, void *scratch, int2 *out, cudaStream_t s)
{
    if (c < 1 || c > 13)
        return cudaErrorInvalidValue;
    if (n == 0)
        return cudaSuccess;
    const uint64_t bins = (uint64_t(1) << (2 * c)) + 1;
    unsigned long long *cnt = static_cast<unsigned long long *>(scratch);
    unsigned long long *part = cnt + bins;
    cudaError_t e = cudaMemsetAsync(cnt, 0, bins * 8, s);
    if (e != cudaSuccess)
        return e;
    const unsigned grid = unsigned(std::min<uint64_t>((n + 255) / 256, uint64_t(device_sm_count()) * 16));
    k_cell_hist<<<grid, 256, 0, s>>>(pts, n, c, cnt);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    if ((e = launch_scan(cnt, bins, nullptr, part, s)) != cudaSuccess) // cnt: cell starts (cursors)
        return e;
    k_cell_scatter<<<grid, 256, 0, s>>>(pts, n, c, cnt, out);
    return cudaGetLastError();
}

uint32_t join_chunk_points() { return kWChunk; }
// part: the bitmap of pass 1 (8 words per chunk = 4 u64), then the scan's partials
uint64_t join_part_words(uint64_t n)
{
    const uint64_t nchunks = (n + kWChunk - 1) / kWChunk;
    return nchunks * (kWItems / 2) + scan_partials(nchunks) + 2;
}

// Passes 1 and 2.  ev (or null): events recorded after pass 1a, after pass 1b
// and after the scan.
static cudaError_t join_resolve_scan(const JoinLaunch &a, unsigned long long *part, cudaStream_t s, cudaEvent_t *ev)
{
    const uint64_t nchunks = (a.n + kWChunk - 1) / kWChunk;
    if (nchunks >= (1ull << 31))
        return cudaErrorInvalidValue;
    if (reinterpret_cast<uintptr_t>(a.pts) & 15)
        return cudaErrorMisalignedAddress;
    if (nchunks == 0)
        return a.total ? cudaMemsetAsync(a.total, 0, sizeof(unsigned long long), s) : cudaSuccess;
    uint32_t *pend = reinterpret_cast<uint32_t *>(part);
    cudaError_t e = launch_pass1(a, pend, s, ev ? ev[0] : nullptr, false);
    if (e != cudaSuccess)
        return e;
    if (ev)
        cudaEventRecord(ev[1], s);
    e = launch_scan(a.tile_tot, nchunks, a.total, part + nchunks * (kWItems / 2), s);
    if (ev)
        cudaEventRecord(ev[2], s);
    return e;
}

cudaError_t launch_join_resolve(const JoinLaunch &a, unsigned long long *part, cudaStream_t s)
{
    return join_resolve_scan(a, part, s, nullptr);
}

cudaError_t launch_join_emit(const JoinLaunch &a, cudaStream_t s, const uint32_t *pend)
{
    const uint32_t nchunks = uint32_t((a.n + kWChunk - 1) / kWChunk);
    if (nchunks == 0 || a.cap == 0)
        return cudaSuccess;
    if (a.narrow && !pend)
        return cudaErrorInvalidValue;
    const uint32_t nblk = (nchunks + kWarps - 1) / kWarps;
    static bool done[12][64] = {};
    return with_switches(a, [&](auto fp32, auto kind) -> cudaError_t {
        constexpr bool F = decltype(fp32)::value;
        constexpr int N = decltype(kind)::value;
        auto kn = k_wemit16<F, false, N>;
        auto kw = k_wemit<F, N>;
        const cudaError_t e = a.narrow ? smem_opt_in(kn, kEmit16Smem<N>, done[F + 2 * N])
                                       : smem_opt_in(kw, kEmitSmem, done[6 + F + 2 * N]);
        if (e != cudaSuccess)
            return e;
        if (a.narrow)
            kn<<<persistent_grid(kn, kThreads, kEmit16Smem<N>, nblk), kThreads, kEmit16Smem<N>, s>>>(a, a.tile_tot, nchunks, pend);
        else
            kw<<<persistent_grid(kw, kThreads, kEmitSmem, nblk), kThreads, kEmitSmem, s>>>(a, a.tile_tot, nchunks);
        return cudaGetLastError();
    });
}

// The join of a small table (at most kSmallChunks chunks, 16-bit results, with an
// output): two
// launches, k_small and k_wemit16<SELF>.  ev as for launch_join.
template <bool FP32, int KIND>
static cudaError_t launch_small(const JoinLaunch &a, uint32_t *pend, cudaStream_t s, cudaEvent_t *ev)
{
    static bool done[64] = {};
    const uint32_t nchunks = uint32_t((a.n + kWChunk - 1) / kWChunk), nblk = (nchunks + kWarps - 1) / kWarps;
    if (ev)
        cudaEventRecord(ev[0], s);
    cudaError_t e = cudaSuccess;
    if (KIND == kDisk && a.ix.P > kDiskSplit) {
        e = launch_disk_pass1<kOut16>(a, pend, s);
    } else {
        k_small<FP32, kOut16, KIND><<<nblk, kThreads, 0, s>>>(a, pend, nchunks, a.ix.P <= kSmallHist ? 1 : 0);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = smem_opt_in(k_wemit16<FP32, true, KIND>, kEmit16Smem<KIND>, done);
    if (e != cudaSuccess)
        return e;
    for (int k = 1; ev && k < 4; ++k)
        cudaEventRecord(ev[k], s);
    k_wemit16<FP32, true, KIND><<<nblk, kThreads, kEmit16Smem<KIND>, s>>>(a, a.tile_tot, nchunks, pend);
    return cudaGetLastError();
}

__global__ void k_sum_u64(unsigned long long *dst, const unsigned long long *x, const unsigned long long *y)
{
    *dst = *x + *y;
}

cudaError_t launch_sum_u64(unsigned long long *dst, const unsigned long long *x, const unsigned long long *y,
                           cudaStream_t s)
{
    k_sum_u64<<<1, 1, 0, s>>>(dst, x, y);
    return cudaGetLastError();
}

// ------------------------------------------------------ local edge lists
// A fine cell of side S at (x0, y0) and the row list of one of its polygons.  An
// edge takes part in the cell's tests through its part over the integer rows
// [y0, y0 + S - 1], and that part is, for the cell's points,
//   left   never crossed by a rightward ray: dropped;
//   right  crossed by every ray of a row it straddles, whatever the point's x:
//          only the parity of such edges per row matters, a step function of y;
//   near   neither for certain: kept.
// (edge_side; in doubt, near.)  The step function is written as edges
// at x = 2^30, right of every point: one over all rows when it is odd at y0, and
// one from t up for every y = t where it changes.  A vertex between two right
// edges changes it twice, so the changes are the few vertices where a chain
// passes from right to near or left.
constexpr uint32_t kLocalMin = 8;   // shorter lists stay
// Mean edges per list from which an index gets local lists.  50M points x 2000 cells,
// without and with: at a mean of 4.2 the join takes 307 / 302 us, the build 4.0 / 4.7
// ms and the index 463 / 519 MB; at 7.7 434 / 387 us, 1.6 / 2.1 ms, 66 / 86 MB; at
// 11.1 627 / 491 us, 1.2 / 1.8 ms, 36 / 55 MB.  Shorter lists repay the build and the
// memory only over many joins, so the line lies above the automatic grids' lists of
// a map of small polygons.
constexpr uint32_t kLocalMean = 8;
constexpr int kLocalTurns = 8;      // changes of parity a cell may record; else the list stays

// The parity of the right edges over the rows of a cell: at y0 (odd), and the y
// where it changes.  add() is false when there are more changes than fit.
struct LocalTurns {
    int turn[kLocalTurns];
    int nt = 0;
    uint32_t odd = 0;

    __device__ __forceinline__ bool add(const int4 &v, const CellBox &c)
    {
        odd ^= (v.y > c.y0) != (v.w > c.y0) ? 1u : 0u;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int y = h ? v.w : v.y;
            if (y <= c.y0 || y >= c.y0 + c.S)
                continue;
            int at = -1;
            for (int i = 0; i < nt; ++i)
                at = turn[i] == y ? i : at;
            if (at >= 0)
                turn[at] = turn[--nt];
            else if (nt < kLocalTurns)
                turn[nt++] = y;
            else
                return false;
        }
        return true;
    }
};

// The long lists and their cells: x entry, y and z the cell's corner, w what
// k_local_size finds (kLocalChanged | changes << 27 | parity << 26 | kept edges; 0: stays).
// Few cells hold one, and seldom two lanes of a warp, so the lists are gathered
// first and then taken a lane each, four edges loaded at a time: 256 queries at
// g = 13 take 1.5 (gathering) + 3.9 + 3.7 ms; with the lists walked where they were
// found, a lane per cell, counting and writing took 4.8 + 12.4 ms.
constexpr uint32_t kLocalChanged = 1u << 31;
constexpr uint32_t kLocalMaxList = 1u << 26;

__device__ __forceinline__ bool local_takes(const uint4 &en)
{
    return (en.w & kEntBoundary) && en.z >= kLocalMin && en.z < kLocalMaxList;
}

// Edges k .. k + kLocalLoads - 1 of the list (past its end, the last one).
constexpr uint32_t kLocalLoads = 4;

__device__ __forceinline__ void load_list(const IndexView &ix, const uint4 &en, uint32_t k, int4 (&v)[kLocalLoads])
{
#pragma unroll
    for (uint32_t u = 0; u < kLocalLoads; ++u)
        v[u] = ix.edge[en.y + min(k + u, en.z - 1)];
}

// A lane per fine cell; *n_items counts (zeroed), in no particular order.
__global__ void __launch_bounds__(256) k_local_items(IndexView ix, const uint32_t *blk_cell, uint64_t n_words, const uint4 *ent,
                                                     unsigned long long *n_items, uint64_t cap, uint4 *items)
{
    const int lane = threadIdx.x & 31;
    for (uint64_t t0 = (uint64_t)blockIdx.x * 256 + (threadIdx.x & ~31u); t0 < n_words; t0 += (uint64_t)gridDim.x * 256) {
        const uint64_t t = t0 + lane;
        const uint32_t w = t < n_words ? ix.fine[t] : 0u;
        const bool lst = (w >> 30) == kCellList;
        uint32_t mine = 0;
        bool more = lst;
        for (uint64_t e = w & kPayloadMask; more; ++e) {
            const uint4 en = ent[e];
            mine += local_takes(en) ? 1u : 0u;
            more = !(en.w & kEntLast);
        }
        if (!__any_sync(kFull, mine != 0))
            continue;
        uint32_t inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(kFull, inc, o);
            inc += lane >= o ? v : 0u;
        }
        unsigned long long at = 0;
        if (lane == 31)
            at = atomicAdd(n_items, (unsigned long long)inc);
        at = __shfl_sync(kFull, at, 31) + (inc - mine);
        if (!mine)
            continue;
        const uint32_t cw = blk_cell[t >> (2 * ix.sb)], f = (uint32_t)t & ((1u << (2 * ix.sb)) - 1);
        const uint32_t x0 = ((cw & ((1u << ix.gc) - 1)) << ix.sc) | ((f & ((1u << ix.sb) - 1)) << ix.sf);
        const uint32_t y0 = ((cw >> ix.gc) << ix.sc) | ((f >> ix.sb) << ix.sf);
        more = true;
        for (uint64_t e = w & kPayloadMask; more; ++e) {
            const uint4 en = ent[e];
            more = !(en.w & kEntLast);
            if (local_takes(en) && at < cap)
                items[at++] = make_uint4((uint32_t)e, x0, y0, 0u);
        }
    }
}

// A lane per long list: items[].w, and totals[0..1] += local edges, changed lists.
__global__ void __launch_bounds__(256) k_local_size(IndexView ix, const uint4 *ent, uint64_t n, uint4 *items,
                                                    unsigned long long *totals)
{
    unsigned long long all_loc = 0, all_ent = 0;
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (uint64_t)gridDim.x * 256) {
        const uint4 it = items[i];
        const uint4 en = ent[it.x];
        const CellBox c{int(it.y), int(it.z), 1 << ix.sf};
        LocalTurns tn;
        uint32_t near = 0;
        bool fits = true;
        for (uint32_t k = 0; k < en.z && fits; k += kLocalLoads) {
            int4 v[kLocalLoads];
            load_list(ix, en, k, v);
#pragma unroll
            for (uint32_t u = 0; u < kLocalLoads; ++u) {
                const int side = k + u < en.z ? edge_side(v[u], c) : 0;
                near += side == 1 ? 1u : 0u;
                fits = fits && (side != 2 || tn.add(v[u], c));
            }
        }
        const uint32_t size = near + tn.odd + (uint32_t)tn.nt;
        if (fits && size * 4 <= en.z * 3) {
            items[i].w = kLocalChanged | ((uint32_t)tn.nt << 27) | (tn.odd << 26) | near;
            all_loc += size;
            ++all_ent;
        }
    }
    all_loc = warp_sum64(all_loc), all_ent = warp_sum64(all_ent);
    if ((threadIdx.x & 31) == 0 && all_ent) {
        atomicAdd(totals, all_loc);
        atomicAdd(totals + 1, all_ent);
    }
}

// A lane per long list: writes the changed ones and their records, at places that
// each warp takes from totals[0..1] (zeroed), in no particular order.  A list that
// does not come out as k_local_size counted it stays what it was (never seen: the
// two kernels decide alike; the bound keeps every write in the list's own place).
__global__ void __launch_bounds__(256) k_local_write(IndexView ix, uint4 *ent, uint64_t n, const uint4 *items,
                                                     unsigned long long *totals, int4 *loc, uint4 *undo)
{
    const int lane = threadIdx.x & 31;
    for (uint64_t i0 = (uint64_t)blockIdx.x * 256 + (threadIdx.x & ~31u); i0 < n; i0 += (uint64_t)gridDim.x * 256) {
        const uint64_t i = i0 + lane;
        const uint4 it = i < n ? items[i] : make_uint4(0u, 0u, 0u, 0u);
        const bool take = it.w & kLocalChanged;
        const uint32_t nt = (it.w >> 27) & 15u, odd = (it.w >> 26) & 1u;
        const uint32_t size = take ? (it.w & (kLocalMaxList - 1)) + odd + nt : 0u;
        const uint32_t b = __ballot_sync(kFull, take);
        if (!b)
            continue;
        unsigned long long inc = size;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long v = __shfl_up_sync(kFull, inc, o);
            inc += lane >= o ? v : 0ull;
        }
        unsigned long long at_loc = 0, at_ent = 0;
        if (lane == 31) {
            at_loc = atomicAdd(totals, inc);
            at_ent = atomicAdd(totals + 1, (unsigned long long)__popc(b));
        }
        at_loc = __shfl_sync(kFull, at_loc, 31) + inc - size;
        at_ent = __shfl_sync(kFull, at_ent, 31) + __popc(b & lanemask_lt());
        if (!take)
            continue;
        const uint4 en = ent[it.x];
        const CellBox c{int(it.y), int(it.z), 1 << ix.sf};
        LocalTurns tn;
        const uint32_t near = it.w & (kLocalMaxList - 1);
        int4 *d = loc + at_loc + odd + nt;
        uint32_t kept = 0;
        bool fits = true;
        for (uint32_t k = 0; k < en.z; k += kLocalLoads) { // in the list's order: right ends descending
            int4 v[kLocalLoads];
            load_list(ix, en, k, v);
#pragma unroll
            for (uint32_t u = 0; u < kLocalLoads; ++u) {
                const int side = k + u < en.z ? edge_side(v[u], c) : 0;
                if (side == 1) {
                    if (kept < near)
                        d[kept] = v[u];
                    ++kept;
                } else if (side == 2) {
                    fits = fits && tn.add(v[u], c);
                }
            }
        }
        undo[at_ent] = make_uint4(it.x, en.y, en.z, 0u);
        if (!fits || kept != near || tn.odd != odd || (uint32_t)tn.nt != nt)
            continue;
        const int far = int(kBox);
        d = loc + at_loc;
        if (odd)
            *d++ = make_int4(far, c.y0, far, c.y0 + c.S);
        for (uint32_t k = 0; k < nt; ++k)
            *d++ = make_int4(far, tn.turn[k], far, c.y0 + c.S);
        ent[it.x].y = kLocalEdge | (uint32_t)at_loc;
        ent[it.x].z = size;
    }
}

// totals[0..2] += the edges that the entries list, the entries that list any, and
// the long lists among them.
__global__ void __launch_bounds__(256) k_list_edges(const uint4 *ent, uint64_t n, unsigned long long *totals)
{
    unsigned long long z = 0, b = 0, l = 0;
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (uint64_t)gridDim.x * 256) {
        const uint4 en = ent[i];
        const bool bnd = en.w & kEntBoundary;
        z += bnd ? en.z : 0u;
        b += bnd ? 1u : 0u;
        l += local_takes(en) ? 1u : 0u;
    }
    z = warp_sum64(z), b = warp_sum64(b), l = warp_sum64(l);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(totals, z);
        atomicAdd(totals + 1, b);
        atomicAdd(totals + 2, l);
    }
}

// The cell of every block.
__global__ void __launch_bounds__(256) k_blk_cell(uint32_t ncell, const uint32_t *cell, uint32_t *blk_cell)
{
    for (uint32_t c = blockIdx.x * 256 + threadIdx.x; c < ncell; c += gridDim.x * 256)
        if ((cell[c] >> 30) == kCellSub)
            blk_cell[cell[c] & kPayloadMask] = c;
}

cudaError_t build_local_lists(const IndexView &view, uint4 *ent, LocalLists &out, size_t max_bytes, cudaStream_t s,
                              cudaMemPool_t pool)
{
    out = LocalLists{};
    const uint64_t n_blk = view.n_fine >> (2 * view.sb), n_words = n_blk << (2 * view.sb);
    if (!n_words || view.n_edge >= kLocalEdge || view.n_ent >= (1ull << 32))
        return cudaSuccess;
    auto blocks = [](uint64_t n) { return unsigned(std::min<uint64_t>((n + 255) / 256, uint64_t(device_sm_count()) * 32)); };
    const size_t b_blk = (n_blk * 4 + 255) & ~size_t(255);
    void *tmp = nullptr, *tmp2 = nullptr;
    unsigned long long h[6] = {}; // local edges, changed lists, edges, lists, long lists, items
    cudaError_t e = cudaMallocFromPoolAsync(&tmp, b_blk + sizeof(h), pool, s);
    if (e != cudaSuccess) { // the index works without them
        cudaGetLastError();
        return cudaSuccess;
    }
    auto done = [&](cudaError_t err) {
        if (tmp2)
            cudaFreeAsync(tmp2, s);
        cudaFreeAsync(tmp, s);
        if (err != cudaSuccess && out.mem) {
            cudaFreeAsync(out.mem, s);
            out = LocalLists{};
        }
        return err;
    };
    uint32_t *blk_cell = static_cast<uint32_t *>(tmp);
    auto *totals = reinterpret_cast<unsigned long long *>(static_cast<char *>(tmp) + b_blk);
    auto read = [&](int n) {
        const cudaError_t x = cudaMemcpyAsync(h, totals, n * 8, cudaMemcpyDeviceToHost, s);
        return x != cudaSuccess ? x : cudaStreamSynchronize(s);
    };
    if ((e = cudaMemsetAsync(totals, 0, sizeof(h), s)) != cudaSuccess)
        return done(e);
    k_list_edges<<<blocks(view.n_ent), 256, 0, s>>>(ent, view.n_ent, totals + 2);
    if ((e = cudaGetLastError()) != cudaSuccess || (e = read(5)) != cudaSuccess)
        return done(e);
    // Maps of 500 to 5000 cells with about 500 vertices each list four edges on
    // average, queries of up to 5000 vertices 40 and 40000 cells of up to 10000
    // vertices 15: the walk of 500M points x 256 queries 4.39 -> 2.74 ms.
    if (h[2] < kLocalMean * h[3] || !h[4])
        return done(cudaSuccess);
    if (cudaMallocFromPoolAsync(&tmp2, h[4] * 16, pool, s) != cudaSuccess) {
        tmp2 = nullptr;
        cudaGetLastError();
        return done(cudaSuccess);
    }
    uint4 *items = static_cast<uint4 *>(tmp2);
    const uint64_t cap = h[4];
    const uint32_t ncell = 1u << (2 * view.gc);
    k_blk_cell<<<blocks(ncell), 256, 0, s>>>(ncell, view.cell, blk_cell);
    k_local_items<<<blocks(n_words), 256, 0, s>>>(view, blk_cell, n_words, ent, totals + 5, cap, items);
    if ((e = cudaGetLastError()) != cudaSuccess || (e = read(6)) != cudaSuccess)
        return done(e);
    const uint64_t n_items = std::min<uint64_t>(h[5], cap);
    if (!n_items)
        return done(cudaSuccess);
    k_local_size<<<blocks(n_items), 256, 0, s>>>(view, ent, n_items, items, totals);
    if ((e = cudaGetLastError()) != cudaSuccess || (e = read(2)) != cudaSuccess)
        return done(e);
    if (h[0] >= kLocalEdge || !h[1])
        return done(cudaSuccess);
    out.bytes = (h[0] + h[1] + 1) * 16;
    if (out.bytes > max_bytes) {
        out = LocalLists{};
        return done(cudaSuccess);
    }
    if (cudaMallocFromPoolAsync(&out.mem, out.bytes, pool, s) != cudaSuccess) {
        out = LocalLists{};
        cudaGetLastError();
        return done(cudaSuccess);
    }
    int4 *loc = static_cast<int4 *>(out.mem);
    uint4 *undo = reinterpret_cast<uint4 *>(loc + h[0]);
    out.loc = loc;
    out.undo = undo;
    out.n_loc = h[0];
    out.n_undo = h[1];
    if ((e = cudaMemsetAsync(totals, 0, 16, s)) != cudaSuccess)
        return done(e);
    k_local_write<<<blocks(n_items), 256, 0, s>>>(view, ent, n_items, items, totals, loc, undo);
    if ((e = cudaGetLastError()) != cudaSuccess || (e = cudaStreamSynchronize(s)) != cudaSuccess)
        return done(e);
    return done(cudaSuccess);
}

int device_sm_count()
{
    int dev = 0;
    cudaGetDevice(&dev);
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n;
}

size_t join_scratch_bytes(uint64_t n)
{
    // per-point results | per-chunk totals (then offsets) | scan partials
    const uint64_t nchunks = (n + kWChunk - 1) / kWChunk;
    return size_t(((n * 4 + 15) & ~uint64_t(15)) + (nchunks + join_part_words(n)) * 8 + 16);
}

size_t plain_scratch_bytes(uint64_t n)
{
    const uint64_t nb = (n + kPlainThreads - 1) / kPlainThreads;
    return size_t(nb * 8 + 16);
}

// The join's scratch: per-point results | per-chunk totals (then offsets) |
// row bitmap and scan partials.  Fills b's result and total pointers and the
// result width.
static unsigned long long *join_layout(JoinLaunch &b, void *scratch)
{
    char *sc = static_cast<char *>(scratch);
    b.res = reinterpret_cast<uint32_t *>(sc);
    b.tile_tot = reinterpret_cast<unsigned long long *>(sc + ((b.n * 4 + 15) & ~uint64_t(15)));
    // 16-bit results when every polygon id and every point's polygon count
    // fit (the row bitmap in part stays in place until pass 3)
    b.narrow = b.ix.P <= kRes16MaxP ? 1 : 0;
    b.aux_bits = 8;
    while ((1u << b.aux_bits) < b.ix.P && b.aux_bits < 16)
        ++b.aux_bits;
    return b.tile_tot + (b.n + kWChunk - 1) / kWChunk;
}

cudaError_t launch_join_count(const JoinLaunch &a, void *scratch, cudaStream_t s, cudaEvent_t *ev)
{
    if ((a.n + kWChunk - 1) / kWChunk >= (1ull << 31))
        return cudaErrorInvalidValue;
    JoinLaunch b = a;
    unsigned long long *part = join_layout(b, scratch);
    cudaError_t e;
    if (a.counts && a.ix.P && !a.keep_counts)
        if ((e = cudaMemsetAsync(a.counts, 0, sizeof(unsigned long long) * a.ix.P, s)) != cudaSuccess)
            return e;
    if (a.n == 0)
        return a.total ? cudaMemsetAsync(a.total, 0, sizeof(unsigned long long), s) : cudaSuccess;
    // passes 1 and 2: resolve every point (counts per polygon, per-point
    // results, per-chunk totals), then the offsets and the total
    if (ev)
        cudaEventRecord(ev[0], s);
    return join_resolve_scan(b, part, s, ev ? ev + 1 : nullptr);
}

cudaError_t launch_join_write(const JoinLaunch &a, void *scratch, cudaStream_t s)
{
    if (a.n == 0)
        return cudaSuccess;
    JoinLaunch b = a;
    unsigned long long *part = join_layout(b, scratch);
    // pass 3: pairs in point order
    return launch_join_emit(b, s, reinterpret_cast<const uint32_t *>(part));
}

cudaError_t launch_join(const JoinLaunch &a, void *scratch, cudaStream_t s, cudaEvent_t *ev)
{
    cudaError_t e;
    if (a.n && (a.n + kWChunk - 1) / kWChunk <= kSmallChunks && a.cap && !a.pair_base && a.ix.P <= kRes16MaxP) {
        if (reinterpret_cast<uintptr_t>(a.pts) & 15)
            return cudaErrorMisalignedAddress;
        JoinLaunch b = a;
        uint32_t *pend = reinterpret_cast<uint32_t *>(join_layout(b, scratch));
        if (a.counts && a.ix.P && !a.keep_counts)
            if ((e = cudaMemsetAsync(a.counts, 0, sizeof(unsigned long long) * a.ix.P, s)) != cudaSuccess)
                return e;
        e = with_switches(b, [&](auto fp32, auto kind) {
            constexpr bool F = decltype(fp32)::value;
        constexpr int N = decltype(kind)::value;
            return launch_small<F, N>(b, pend, s, ev);
        });
        if (ev)
            cudaEventRecord(ev[4], s);
        return e;
    }
    e = launch_join_count(a, scratch, s, ev);
    if (e != cudaSuccess || a.n == 0)
        return e;
    if ((e = launch_join_write(a, scratch, s)) != cudaSuccess)
        return e;
    if (ev)
        cudaEventRecord(ev[4], s);
    return cudaSuccess;
}

bool use_directory(const JoinLaunch &a)
{
    return a.clustered && a.cell_end && a.cluster_log2 >= a.ix.gc && a.cluster_log2 <= 13 && !a.near.any();
}

// A table in row order is counted by the join's pass 1 with nothing kept but the
// row bitmap: the points of blocks that the summary resolves read no index
// word, and the exact tests run in their own kernel instead of holding up the
// streaming warps (100M points: 5000-cell map 1928 -> 530 us, 2000 cells 883 ->
// 345, 64 queries 1020 -> 409, 256 stars 478 -> 305).  From 2M points on: at 2M
// two launches cost as much as they save (2000 cells 25.8 one pass / 28.9, at 4M
// 50.9 / 38.1).  Only with the summary: without it (a 40000-cell map, counts in
// global memory) the one pass is as fast (2021 / 2068 us).
constexpr uint64_t kSplitCountMin = uint64_t(1) << 21;
// A disk index's one pass (k_disk_pass1) holds out longer: 2.5M points x 64 / 1024 disks
// 14.5 / 19.6 us in one, 21.1 / 26.1 in two, 6M 23.0 / 33.2 and 25.8 / 31.4, 20M 54 / 77
// and 46 / 61, 100M 231 / 333 and 155 / 234.
constexpr uint64_t kDiskSplitCountMin = uint64_t(1) << 23;
bool use_split_count(const JoinLaunch &a)
{
    if (a.near.disk)
        return a.n > kDiskSplitCountMin && !a.clustered && a.ix.use_sum && a.ix.P <= kDiskSplit;
    return a.n > kSplitCountMin && (a.near.rad || (!a.clustered && a.ix.use_sum));
}

static size_t split_count_bytes(uint64_t n)
{
    return n > kSplitCountMin ? size_t((n + kWChunk - 1) / kWChunk) * kWItems * 4 : 0;
}

size_t aggregate_scratch_bytes(const JoinLaunch &a)
{
    return use_directory(a)                 ? size_t((a.n + kWChunk - 1) / kWChunk) * kWItems * 4
           : !a.clustered || a.near.rad ? split_count_bytes(a.n)
                                        : 0;
}

cudaError_t launch_aggregate(const JoinLaunch &a, void *scratch, cudaStream_t s, cudaEvent_t *ev)
{
    cudaError_t e = cudaSuccess;
    if (!a.keep_counts)
        e = cudaMemsetAsync(a.counts, 0, sizeof(unsigned long long) * (a.ix.P ? a.ix.P : 1), s);
    if (e != cudaSuccess || a.n == 0)
        return e;
    if (reinterpret_cast<uintptr_t>(a.pts) & 15)
        return cudaErrorMisalignedAddress;
    if (scratch && use_split_count(a)) {
        if (ev)
            cudaEventRecord(ev[0], s);
        uint32_t *pend = static_cast<uint32_t *>(scratch);
        e = launch_pass1(a, pend, s, nullptr, true);
        if (ev)
            cudaEventRecord(ev[1], s);
        return e;
    }
    if (a.near.disk)
        return launch_pass1(a, nullptr, s, nullptr, true);
    if (a.near.any()) { // few points, or no scratch to have: one launch that keeps nothing
        const uint64_t nchunks = (a.n + kWChunk - 1) / kWChunk;
        if (a.n >= (1ull << 32))
            return cudaErrorInvalidValue;
        const unsigned nblk = unsigned((nchunks + kWarps - 1) / kWarps);
        const int hist = a.ix.P <= kSmallHist ? 1 : 0;
        return with_switches(a, [&](auto fp32, auto kind) {
            if constexpr (decltype(kind)::value == kNear)
                k_small<decltype(fp32)::value, kOutCount, decltype(kind)::value>
                    <<<nblk, kThreads, 0, s>>>(a, nullptr, uint32_t(nchunks), hist);
            return cudaGetLastError();
        });
    }
    const int use_hist = a.ix.P <= (uint32_t)kHistMax ? 1 : 0;
    if (ev)
        cudaEventRecord(ev[0], s);
    if (use_directory(a) && scratch) {
        // cells INSIDE one polygon counted from the directory, then the rows of mixed cells
        uint32_t *rows = static_cast<uint32_t *>(scratch);
        if ((e = cudaMemsetAsync(rows, 0, aggregate_scratch_bytes(a), s)) != cudaSuccess)
            return e;
        const uint32_t side = 1u << a.cluster_log2, units = ((side + 31) / 32) * ((side + kDirRows - 1) / kDirRows);
        const unsigned grid = std::min((units + 7) / 8, uint32_t(device_sm_count()) * 8);
        k_agg_cells<<<grid, 256, 0, s>>>(a.cell_end, a.cluster_log2, a.ix, a.counts, rows, a.stats);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return e;
        e = a.fp32 ? launch_walk<true, kOutCount, kPoly, true>(a, rows, s)
                   : launch_walk<false, kOutCount, kPoly, true>(a, rows, s);
    } else if (a.clustered)
        e = a.fp32 ? launch_warp_kernel<true, true>(a, use_hist, s) : launch_warp_kernel<false, true>(a, use_hist, s);
    else
        e = a.fp32 ? launch_warp_kernel<true, false>(a, use_hist, s) : launch_warp_kernel<false, false>(a, use_hist, s);
    if (ev)
        cudaEventRecord(ev[1], s);
    return e;
}

size_t select_scratch_bytes(uint64_t n, uint32_t P, uint64_t cap, bool aux)
{
    return ((join_scratch_bytes(n) + 15) & ~size_t(15)) + (aux ? n * 8 : 0) + 16 + cap * 8 + partition_scratch_bytes(cap, P);
}

size_t partition_scratch_bytes(uint64_t cap, uint32_t P)
{
    // super_tile leaves fewer than 2 kSuperTiles tiles, or takes the largest or the
    // smallest size; this bound, unlike the count itself, grows with cap
    const uint64_t n_super = std::max((cap + kSuperTileMax - 1) / kSuperTileMax,
                                      std::min<uint64_t>((cap + kSuperTileMin - 1) / kSuperTileMin, 2 * kSuperTiles));
    const uint64_t tab = uint64_t(P) * (n_super ? n_super : 1);
    return size_t(tab * 8 + (scan_partials(tab) + 2) * 8 + 64);
}

cudaError_t launch_partition(const uint2 *pairs, const unsigned long long *total, uint64_t cap, uint32_t P,
                             uint32_t *ids, unsigned long long *offsets, void *scratch, cudaStream_t s)
{
    if (P > (uint32_t)kSelMaxQ)
        return cudaErrorInvalidValue;
    const uint32_t tile = super_tile(cap);
    const uint64_t n_super64 = (cap + tile - 1) / tile;
    if (n_super64 >= (1ull << 31))
        return cudaErrorInvalidValue;
    if (P == 0)
        return cudaMemsetAsync(offsets, 0, sizeof(unsigned long long), s);
    const uint32_t n_super = uint32_t(n_super64 ? n_super64 : 1);
    unsigned long long *table = static_cast<unsigned long long *>(scratch);
    unsigned long long *part = table + uint64_t(P) * n_super;
    unsigned long long *tab_total = part + scan_partials(uint64_t(P) * n_super) + 1;
    // per (query, super-tile) counts of the pairs, scanned in query-major order
    k_part_count<<<n_super, kThreads, sizeof(uint32_t) * P, s>>>(pairs, total, cap, P, table, n_super, tile);
    cudaError_t e = launch_scan(table, uint64_t(P) * n_super, tab_total, part, s);
    if (e != cudaSuccess)
        return e;
    k_sel_offsets<<<(P + 256) / 256, 256, 0, s>>>(table, n_super, P, total, offsets);
    // point ids, ascending per query
    static bool done[64] = {};
    if ((e = smem_opt_in(k_part_emit, part_smem(kSelMaxQ), done)) != cudaSuccess)
        return e;
    if (cap)
        k_part_emit<<<n_super, kThreads, part_smem(P), s>>>(pairs, total, P, table, n_super, ids, cap, tile);
    return cudaGetLastError();
}

cudaError_t launch_select(const JoinLaunch &a, uint32_t *ids, uint64_t cap, unsigned long long *offsets,
                          void *scratch, cudaStream_t s, bool with_aux)
{
    if (a.ix.P > (uint32_t)kSelMaxQ)
        return cudaErrorInvalidValue;
    char *sc = static_cast<char *>(scratch);
    void *join_scratch = sc;
    sc += (join_scratch_bytes(a.n) + 15) & ~size_t(15);
    // overlapping queries put many points in several polygons: pass 1b packs
    // their ids (in the scratch, or where the caller says) so that pass 3 does not
    // walk them again
    uint64_t *aux = with_aux ? reinterpret_cast<uint64_t *>(sc) : a.aux;
    sc += with_aux ? a.n * 8 : 0;
    unsigned long long *total = reinterpret_cast<unsigned long long *>(sc);
    sc += 16;
    uint2 *pairs = reinterpret_cast<uint2 *>(sc);
    sc += cap * 8;
    // 1. the join: (point, query) pairs in point order, and their total
    JoinLaunch b = a;
    b.pairs = pairs;
    b.cap = cap;
    b.counts = nullptr;
    b.total = total;
    b.aux = aux;
    cudaError_t e = launch_join(b, join_scratch, s);
    if (e != cudaSuccess)
        return e;
    // 2. stable partition by query
    return launch_partition(pairs, total, cap, a.ix.P, ids, offsets, sc, s);
}

cudaError_t launch_join_plain(const JoinLaunch &a, void *scratch, cudaStream_t s)
{
    const uint64_t nb = (a.n + kPlainThreads - 1) / kPlainThreads;
    if (nb >= (1ull << 31))
        return cudaErrorInvalidValue;
    unsigned long long *block = reinterpret_cast<unsigned long long *>(scratch);
    cudaError_t e;
    if (a.counts && a.ix.P) {
        e = cudaMemsetAsync(a.counts, 0, sizeof(unsigned long long) * a.ix.P, s);
        if (e != cudaSuccess)
            return e;
    }
    if (nb == 0) {
        if (a.total)
            return cudaMemsetAsync(a.total, 0, sizeof(unsigned long long), s);
        return cudaSuccess;
    }
    k_plain_count<<<(unsigned)nb, kPlainThreads, 0, s>>>(a, block);
    k_scan<<<1, 1024, 0, s>>>(block, nb, a.total);
    k_plain_write<<<(unsigned)nb, kPlainThreads, 0, s>>>(a, block);
    return cudaGetLastError();
}

// ------------------------------------------------------ multi-request launchers
namespace {
uint64_t multi_ntiles(uint64_t n) { return (n + kMChunk - 1) / kMChunk; }
uint64_t multi_part_words(uint64_t ntiles) { return scan_partials(ntiles) + 2; }
} // namespace

size_t multi_scratch_bytes(uint64_t n, int K)
{
    const uint64_t nt = multi_ntiles(n);
    return size_t(K) * size_t(nt + multi_part_words(nt)) * 8 + 256;
}

static cudaError_t multi_check(const MultiLaunch &m)
{
    if (m.K < 1 || m.K > kMaxBatch)
        return cudaErrorInvalidValue;
    if (reinterpret_cast<uintptr_t>(m.pts) & 7)
        return cudaErrorMisalignedAddress;
    if (multi_ntiles(m.n) >= (1ull << 31))
        return cudaErrorInvalidValue;
    return cudaSuccess;
}

cudaError_t launch_multi_count(const MultiLaunch &m, void *scratch, cudaStream_t s)
{
    cudaError_t e = multi_check(m);
    if (e != cudaSuccess)
        return e;
    for (int r = 0; r < m.K; ++r)
        if (m.counts[r] && m.ix[r].P)
            if ((e = cudaMemsetAsync(m.counts[r], 0, sizeof(unsigned long long) * m.ix[r].P, s)) != cudaSuccess)
                return e;
    const uint64_t nt = multi_ntiles(m.n);
    if (nt == 0)
        return cudaMemsetAsync(m.totals, 0, sizeof(unsigned long long) * m.K, s);
    unsigned long long *tile_tot = static_cast<unsigned long long *>(scratch);
    unsigned long long *part = tile_tot + uint64_t(m.K) * nt;
    const int use_hist = m.qbase[m.K] <= kMultiHistMax ? 1 : 0;
    const size_t smem = kMultiSmem + (use_hist ? sizeof(uint32_t) * m.qbase[m.K] : 0);
    static bool done[2][64] = {};
    if (m.fp32) {
        if ((e = smem_opt_in(k_multi<true, false>, kMultiSmem + 4 * kMultiHistMax, done[0])) != cudaSuccess)
            return e;
        k_multi<true, false><<<persistent_grid(k_multi<true, false>, kThreads, smem, uint32_t((nt + kWarps - 1) / kWarps)), kThreads, smem,
                               s>>>(m, tile_tot, uint32_t(nt), use_hist);
    } else {
        if ((e = smem_opt_in(k_multi<false, false>, kMultiSmem + 4 * kMultiHistMax, done[1])) != cudaSuccess)
            return e;
        k_multi<false, false><<<persistent_grid(k_multi<false, false>, kThreads, smem, uint32_t((nt + kWarps - 1) / kWarps)), kThreads,
                                smem, s>>>(m, tile_tot, uint32_t(nt), use_hist);
    }
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    for (int r = 0; r < m.K; ++r)
        if ((e = launch_scan(tile_tot + uint64_t(r) * nt, nt, m.totals + r, part + uint64_t(r) * multi_part_words(nt),
                             s)) != cudaSuccess)
            return e;
    return cudaSuccess;
}

cudaError_t launch_multi_emit(const MultiLaunch &m, void *scratch, cudaStream_t s)
{
    cudaError_t e = multi_check(m);
    if (e != cudaSuccess)
        return e;
    const uint64_t nt = multi_ntiles(m.n);
    if (nt == 0)
        return cudaSuccess;
    unsigned long long *tile_tot = static_cast<unsigned long long *>(scratch);
    const size_t smem = kMultiSmem;
    static bool done[2][64] = {};
    const size_t smem_max = kMultiSmem;
    if (m.fp32) {
        if ((e = smem_opt_in(k_multi<true, true>, smem_max, done[0])) != cudaSuccess)
            return e;
        k_multi<true, true><<<persistent_grid(k_multi<true, true>, kThreads, smem, uint32_t((nt + kWarps - 1) / kWarps)), kThreads, smem,
                              s>>>(m, tile_tot, uint32_t(nt), 0);
    } else {
        if ((e = smem_opt_in(k_multi<false, true>, smem_max, done[1])) != cudaSuccess)
            return e;
        k_multi<false, true><<<persistent_grid(k_multi<false, true>, kThreads, smem, uint32_t((nt + kWarps - 1) / kWarps)), kThreads, smem,
                               s>>>(m, tile_tot, uint32_t(nt), 0);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------ plain path in two halves (serving comparison)
size_t plain_split_scratch_bytes(uint64_t n)
{
    const uint64_t nb = (n + kPlainThreads - 1) / kPlainThreads;
    return size_t(nb + scan_partials(nb) + 2) * 8 + 64;
}

cudaError_t launch_plain_count(const JoinLaunch &a, void *scratch, cudaStream_t s)
{
    const uint64_t nb = (a.n + kPlainThreads - 1) / kPlainThreads;
    if (nb >= (1ull << 31))
        return cudaErrorInvalidValue;
    cudaError_t e;
    if (a.counts && a.ix.P)
        if ((e = cudaMemsetAsync(a.counts, 0, sizeof(unsigned long long) * a.ix.P, s)) != cudaSuccess)
            return e;
    if (nb == 0)
        return cudaMemsetAsync(a.total, 0, sizeof(unsigned long long), s);
    unsigned long long *block = static_cast<unsigned long long *>(scratch);
    k_plain_count<<<(unsigned)nb, kPlainThreads, 0, s>>>(a, block);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return e;
    return launch_scan(block, nb, a.total, block + nb, s);
}

cudaError_t launch_plain_write(const JoinLaunch &a, void *scratch, cudaStream_t s)
{
    const uint64_t nb = (a.n + kPlainThreads - 1) / kPlainThreads;
    if (nb == 0)
        return cudaSuccess;
    k_plain_write<<<(unsigned)nb, kPlainThreads, 0, s>>>(a, static_cast<const unsigned long long *>(scratch));
    return cudaGetLastError();
}

// ------------------------------------------------ buffered polygons: launchers
// Sets the bits of the cells of a 2^g grid that list items or meet a non-empty
// coarse cell of the polygons' own index (2^gp).
__global__ void k_buf_mask(const uint32_t *cell, int gp, const uint32_t *cell_off, uint32_t *mask, int g)
{
    const uint64_t nc = uint64_t(1) << (2 * g);
    for (uint64_t c = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += (uint64_t)gridDim.x * blockDim.x)
        if (cell_off[c + 1] > cell_off[c])
            atomicOr(mask + (c >> 5), 1u << (c & 31));
    const uint64_t n = uint64_t(1) << (2 * gp);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        if (!cell[i])
            continue;
        const uint32_t cx = uint32_t(i & ((1u << gp) - 1)), cy = uint32_t(i >> gp);
        if (g <= gp) { // one mask cell holds 2^(gp - g) x 2^(gp - g) coarse cells
            const uint32_t m = ((cy >> (gp - g)) << g) | (cx >> (gp - g));
            atomicOr(mask + (m >> 5), 1u << (m & 31));
        } else { // the coarse cell spans 2^(g - gp) x 2^(g - gp) mask cells
            const uint32_t k = 1u << (g - gp);
            for (uint32_t y = cy * k; y < (cy + 1) * k; ++y)
                for (uint32_t x = cx * k; x < (cx + 1) * k; ++x) {
                    const uint32_t m = (y << g) | x;
                    atomicOr(mask + (m >> 5), 1u << (m & 31));
                }
        }
    }
}

static cudaError_t launch_buffer_mask(const IndexView &ix, const uint32_t *cell_off, uint32_t *mask, int g)
{
    const uint64_t n = uint64_t(1) << (2 * ix.gc);
    const unsigned grid = unsigned(std::min<uint64_t>((n + 255) / 256, uint64_t(device_sm_count()) * 32));
    k_buf_mask<<<grid, 256>>>(ix.cell, ix.gc, cell_off, mask, g);
    return cudaGetLastError();
}

// The index of buffered polygons (NearView) from the edge grid.  A cell's groups
// (its polygons, ascending) are the union of the groups of items of its edge-grid
// cell and of the polygons that hold its corner.  With S the side of the cell:
//   whole   every point of the cell meets the polygon: the group is flagged
//           kBufferFull, or one edge has the cell's four extreme points within r
//           (the points within r of a segment are a convex set), or the polygon
//           holds the corner and no edge's box meets the cell;
//   cross   an edge's box meets the cell, so points of the cell may differ in
//           being inside (an edge that passes between two points of the cell is
//           listed there: the listing reaches every edge within r >= 0 of the
//           box of the cell's points);
//   edges   those within r + h + 2 of the cell's centre, h half its diagonal, in
//           FP32 with the coordinate differences' rounding (2^-24 relative, a
//           few of them) covered by 2^-18 of their sum;
//   none    neither cross nor edges: no point of the cell meets the polygon.
// Calls add(q, first item, end, flags) for every group of the cell but those
// that no point meets: flags 0 for whole, else kEntBoundary and kEntCross.
template <class F>
__device__ __forceinline__ void near_groups(const IndexView &in, const uint32_t *item_q, const int4 *item_seg,
                                            const int32_t *rad, uint32_t k, uint32_t kend, const CellBox &c, F add)
{
    const int x1 = c.x0 + c.S - 1, y1 = c.y0 + c.S - 1;
    auto group = [&](uint32_t q, bool holds) {
        const uint32_t k0 = k;
        if (item_q[k] & kBufferFull) {
            ++k;
            add(q, 0u, 0u, 0u);
            return;
        }
        const int r = rad[q];
        bool cross = false, reach = false, whole = false;
        for (; k < kend && item_q[k] == q; ++k) {
            const int4 v = item_seg[k];
            cross = cross || (min(v.x, v.z) <= x1 && max(v.x, v.z) >= c.x0 && min(v.y, v.w) <= y1 && max(v.y, v.w) >= c.y0);
            if (!whole && edge_reaches(v, c, r)) {
                reach = true;
                whole = seg_near<true>(v, c.x0, c.y0, r) && seg_near<true>(v, x1, c.y0, r) &&
                        seg_near<true>(v, c.x0, y1, r) && seg_near<true>(v, x1, y1, r);
            }
        }
        if (whole || (holds && !cross))
            add(q, 0u, 0u, 0u);
        else if (reach || cross)
            add(q, k0, k, kEntBoundary | (cross ? kEntCross : 0u));
    };
    auto inside = [&](uint32_t q) {
        while (k < kend && (item_q[k] & ~kBufferFull) < q)
            group(item_q[k] & ~kBufferFull, false);
        if (k < kend && (item_q[k] & ~kBufferFull) == q)
            group(q, true);
        else
            add(q, 0u, 0u, 0u);
    };
    uint32_t t = 0, s = 0;
    const uint64_t keep = policy_evict_last();
    const uint32_t w = resolve(in, (uint32_t)c.x0, (uint32_t)c.y0, keep);
    if ((w >> 30) == kCellInsideOne)
        inside(w & kPayloadMask);
    else if ((w >> 30) == kCellList)
        walk_entries<false>(in, in.ent + (w & kPayloadMask), c.x0, c.y0, t, s, keep, inside);
    while (k < kend)
        group(item_q[k] & ~kBufferFull, false);
}

// Coarse level, a thread per cell.  COUNT: the cell's word (kinds kCellSub and
// kCellCoarseList without their payload), its entries when it is a coarse list,
// and 1 when it is split.  Else: the payloads and the coarse lists, each within the
// place that was counted for it (*wrong counts those that come out otherwise).
template <bool COUNT>
__global__ void __launch_bounds__(256) k_near_coarse(IndexView in, const uint32_t *cell_off, const uint32_t *item_q,
                                                     const int4 *item_seg, const int32_t *rad, const uint32_t *mask,
                                                     int g, unsigned long long *n_ent, unsigned long long *n_blk,
                                                     uint32_t *cell, uint4 *ent, uint64_t ent_end,
                                                     unsigned long long *wrong)
{
    const uint32_t ncell = 1u << (2 * g);
    const int sh = kBoxLog2 - g;
    for (uint32_t c = blockIdx.x * 256 + threadIdx.x; c < ncell; c += gridDim.x * 256) {
        if (COUNT && !((mask[c >> 5] >> (c & 31)) & 1u)) {
            n_ent[c] = n_blk[c] = 0;
            cell[c] = 0u;
            continue;
        }
        const uint32_t kind = COUNT ? 0u : cell[c] >> 30;
        if (!COUNT && kind < kCellSub)
            continue;
        if (!COUNT && kind == kCellSub) {
            cell[c] |= (uint32_t)n_blk[c];
            continue;
        }
        const CellBox nc{int((c & ((1u << g) - 1)) << sh), int((c >> g) << sh), 1 << sh};
        const uint64_t off = COUNT ? 0 : n_ent[c], room = COUNT ? 0 : (c + 1 < ncell ? n_ent[c + 1] : ent_end) - off;
        uint32_t n = 0, one = 0;
        bool lists = false;
        near_groups(in, item_q, item_seg, rad, cell_off[c], cell_off[c + 1], nc,
                    [&](uint32_t q, uint32_t, uint32_t, uint32_t flags) {
                        if (!COUNT && n < room)
                            ent[off + n] = make_uint4(q, 0u, 0u, n + 1 == room ? kEntLast : 0u);
                        one = q;
                        lists = lists || flags;
                        ++n;
                    });
        if (COUNT) {
            n_ent[c] = !lists && n > 1 ? n : 0;
            n_blk[c] = lists ? 1 : 0;
            cell[c] = lists ? kCellSub << 30 : n > 1 ? kCellCoarseList << 30 : n ? (kCellInsideOne << 30) | one : 0u;
        } else {
            if (n != room || lists)
                atomicAdd(wrong, 1ull);
            cell[c] |= uint32_t(off);
        }
    }
}

// The cell of every block.
__global__ void __launch_bounds__(256) k_near_blocks(uint32_t ncell, const uint32_t *cell,
                                                     const unsigned long long *n_blk, uint32_t *blk_cell)
{
    for (uint32_t c = blockIdx.x * 256 + threadIdx.x; c < ncell; c += gridDim.x * 256)
        if ((cell[c] >> 30) == kCellSub)
            blk_cell[n_blk[c]] = c;
}

// Fine level, a thread per fine cell of every block.  COUNT: its word (a list's
// without its offset), its entries and its edges; else the lists, as above.
template <bool COUNT>
__global__ void __launch_bounds__(256) k_near_fine(IndexView in, const uint32_t *cell_off, const uint32_t *item_q,
                                                   const int4 *item_seg, const int32_t *rad, int g, int sb,
                                                   const uint32_t *blk_cell, uint64_t n_fine, unsigned long long *n_ent,
                                                   unsigned long long *n_edge, uint64_t ent0, uint32_t *fine, uint4 *ent,
                                                   int4 *edge, uint64_t ent_end, uint64_t edge_end,
                                                   unsigned long long *wrong)
{
    const int sh = kBoxLog2 - g, sf = sh - sb;
    const uint32_t fm = (1u << sb) - 1;
    for (uint64_t t = (uint64_t)blockIdx.x * 256 + threadIdx.x; t < n_fine; t += (uint64_t)gridDim.x * 256) {
        if (!COUNT && (fine[t] >> 30) != kCellList)
            continue;
        const uint32_t c = blk_cell[t >> (2 * sb)], f = (uint32_t)t & ((1u << (2 * sb)) - 1);
        const CellBox nc{int(((c & ((1u << g) - 1)) << sh) | ((f & fm) << sf)), int(((c >> g) << sh) | ((f >> sb) << sf)),
                          1 << sf};
        const uint64_t off = COUNT ? 0 : ent0 + n_ent[t], eoff = COUNT ? 0 : n_edge[t];
        const uint64_t room = COUNT ? 0 : (t + 1 < n_fine ? n_ent[t + 1] : ent_end) - n_ent[t];
        const uint64_t eroom = COUNT ? 0 : (t + 1 < n_fine ? n_edge[t + 1] : edge_end) - eoff;
        uint32_t n = 0, one = 0, ne = 0;
        bool whole = false;
        near_groups(in, item_q, item_seg, rad, cell_off[c], cell_off[c + 1], nc,
                    [&](uint32_t q, uint32_t k0, uint32_t k1, uint32_t flags) {
                        const uint32_t first = ne;
                        for (uint32_t k = k0; k < k1; ++k) {
                            const int4 v = item_seg[k];
                            if (edge_reaches(v, nc, rad[q])) {
                                if (!COUNT && ne < eroom)
                                    edge[eoff + ne] = v;
                                ++ne;
                            }
                        }
                        if (!COUNT && n < room)
                            ent[off + n] = make_uint4(q, uint32_t(eoff + first), ne - first,
                                                      flags | (n + 1 == room ? kEntLast : 0u));
                        one = q;
                        whole = !flags;
                        ++n;
                    });
        if (COUNT) {
            const bool lst = n > 1 || (n == 1 && !whole);
            n_ent[t] = lst ? n : 0;
            n_edge[t] = lst ? ne : 0;
            fine[t] = lst ? kCellList << 30 : n ? (kCellInsideOne << 30) | one : 0u;
        } else {
            if (n != room || ne != eroom)
                atomicAdd(wrong, 1ull);
            fine[t] = (kCellList << 30) | uint32_t(off);
        }
    }
}

// Block summary of the coarse words (an empty block, one polygon holding it, or
// mixed), the number of blocks that are not mixed, and (not null) the sentinels.
__global__ void __launch_bounds__(256) k_near_sum(int g, int sg, const uint32_t *cell, uint16_t *sum,
                                                  unsigned long long *resolved, uint4 *ent_end, int4 *edge_end)
{
    const uint32_t nb = 1u << sg, sh = uint32_t(g - sg), t = blockIdx.x * 256 + threadIdx.x;
    if (ent_end && t < 4)
        ent_end[t] = make_uint4(0u, 0u, 0u, kEntLast);
    if (edge_end && t == 0)
        *edge_end = make_int4(0, 0, 0, 0);
    if (t >= nb * nb)
        return;
    const uint32_t by = t / nb, bx = t % nb, w0 = cell[(uint64_t(by << sh) << g) | (bx << sh)];
    bool same = (w0 >> 30) == kCellEmpty || ((w0 >> 30) == kCellInsideOne && (w0 & kPayloadMask) < kSumEmpty);
    for (uint32_t cy = by << sh; same && cy < ((by + 1) << sh); ++cy)
        for (uint32_t cx = bx << sh; same && cx < ((bx + 1) << sh); ++cx)
            same = cell[(uint64_t(cy) << g) | cx] == w0;
    sum[t] = uint16_t(!same ? kSumMixed : (w0 >> 30) == kCellEmpty ? kSumEmpty : (w0 & kPayloadMask));
    if (same)
        atomicAdd(resolved, 1ull);
}

int build_near_index_device(const IndexView &in, const uint32_t *cell_off, const uint32_t *item_q, const int4 *item_seg,
                            const int32_t *rad, int g, NearIndexDev &out, cudaError_t &cerr)
{
    out = NearIndexDev{};
    const uint32_t ncell = 1u << (2 * g);
    const int sg = std::min(g, kSumLog2);
    auto up = [](size_t v) { return (v + 255) & ~size_t(255); };
    char *tmp = nullptr, *tmp2 = nullptr;
    cudaError_t &e = cerr;
    auto done = [&](int status) {
        cudaFree(tmp);
        cudaFree(tmp2);
        if (status && out.mem) {
            cudaFree(out.mem);
            out.mem = nullptr;
        }
        return status;
    };
    auto blocks = [](uint64_t n) { return unsigned(std::min<uint64_t>((n + 255) / 256, uint64_t(device_sm_count()) * 32)); };
    const size_t t_cnt = up(size_t(ncell) * 8), t_part = up((scan_partials(ncell) + 2) * 8),
                 t_mask = up(std::max<size_t>(ncell / 8, 4)), b_cell = up(size_t(ncell) * 4),
                 b_sum = up(std::max<size_t>(size_t(2) << (2 * sg), 16));
    if ((e = cudaMalloc(&tmp, 2 * t_cnt + t_part + t_mask + 2 * b_cell + 256)) != cudaSuccess)
        return done(2);
    auto *n_ent = reinterpret_cast<unsigned long long *>(tmp);
    auto *n_blk = reinterpret_cast<unsigned long long *>(tmp + t_cnt);
    auto *part = reinterpret_cast<unsigned long long *>(tmp + 2 * t_cnt);
    auto *mask = reinterpret_cast<uint32_t *>(tmp + 2 * t_cnt + t_part);
    auto *word = reinterpret_cast<uint32_t *>(tmp + 2 * t_cnt + t_part + t_mask);
    auto *blk_cell = reinterpret_cast<uint32_t *>(tmp + 2 * t_cnt + t_part + t_mask + b_cell);
    // coarse entries, blocks, fine entries, fine edges, resolved summary blocks,
    // lists that the two passes over their cell see differently
    auto *tot = reinterpret_cast<unsigned long long *>(tmp + 2 * t_cnt + t_part + t_mask + 2 * b_cell);
    unsigned long long h[6] = {};
    if ((e = cudaMemset(mask, 0, t_mask)) != cudaSuccess || (e = cudaMemset(tot, 0, sizeof(h))) != cudaSuccess ||
        (e = launch_buffer_mask(in, cell_off, mask, g)) != cudaSuccess)
        return done(2);
    k_near_coarse<true><<<blocks(ncell), 256>>>(in, cell_off, item_q, item_seg, rad, mask, g, n_ent, n_blk, word, nullptr,
                                               0, nullptr);
    if ((e = cudaGetLastError()) != cudaSuccess || (e = launch_scan(n_ent, ncell, tot, part, nullptr)) != cudaSuccess ||
        (e = launch_scan(n_blk, ncell, tot + 1, part, nullptr)) != cudaSuccess ||
        (e = cudaMemcpy(h, tot, 16, cudaMemcpyDeviceToHost)) != cudaSuccess)
        return done(2);
    const uint64_t NB = h[1];
    k_near_blocks<<<blocks(ncell), 256>>>(ncell, word, n_blk, blk_cell);
    // 8 x 8 fine cells per split cell, fewer where that would be more than 2^27
    // fine cells, or more entries or edges than their offsets can name
    for (int sb = kMaxSubLog2;; --sb) {
        const uint64_t nf = NB << (2 * sb);
        if (sb && (nf > (uint64_t(1) << 27) || g + sb > kMaxFineLog2))
            continue;
        const size_t t_f = up(std::max<uint64_t>(nf, 1) * 8), t_fp = up((scan_partials(nf) + 2) * 8),
                     t_fw = up(std::max<uint64_t>(nf, 1) * 4);
        if ((e = cudaMalloc(&tmp2, 2 * t_f + t_fp + t_fw)) != cudaSuccess) {
            if (!sb)
                return done(2);
            cudaGetLastError();
            tmp2 = nullptr;
            continue;
        }
        auto *f_ent = reinterpret_cast<unsigned long long *>(tmp2);
        auto *f_edge = reinterpret_cast<unsigned long long *>(tmp2 + t_f);
        auto *f_part = reinterpret_cast<unsigned long long *>(tmp2 + 2 * t_f);
        auto *f_word = reinterpret_cast<uint32_t *>(tmp2 + 2 * t_f + t_fp);
        if (NB) {
            k_near_fine<true><<<blocks(nf), 256>>>(in, cell_off, item_q, item_seg, rad, g, sb, blk_cell, nf, f_ent, f_edge, 0,
                                                   f_word, nullptr, nullptr, 0, 0, nullptr);
            if ((e = cudaGetLastError()) != cudaSuccess || (e = launch_scan(f_ent, nf, tot + 2, f_part, nullptr)) != cudaSuccess ||
                (e = launch_scan(f_edge, nf, tot + 3, f_part, nullptr)) != cudaSuccess ||
                (e = cudaMemcpy(h, tot, 32, cudaMemcpyDeviceToHost)) != cudaSuccess)
                return done(2);
        }
        if (h[0] + h[2] + 4 > kPayloadMask || h[3] + 1 >= (1ull << 32)) {
            if (!sb)
                return done(1);
            cudaFree(tmp2);
            tmp2 = nullptr;
            continue;
        }
        const size_t b_fine = t_fw, b_ent = up((h[0] + h[2] + 4) * sizeof(uint4)), b_edge = up((h[3] + 1) * sizeof(int4));
        out.bytes = b_cell + b_fine + b_ent + b_edge + b_sum;
        if ((e = cudaMalloc(&out.mem, out.bytes)) != cudaSuccess) {
            out.mem = nullptr;
            if (!sb)
                return done(2);
            cudaGetLastError();
            cudaFree(tmp2);
            tmp2 = nullptr;
            continue;
        }
        char *m = static_cast<char *>(out.mem);
        out.cell = reinterpret_cast<uint32_t *>(m);
        out.fine = reinterpret_cast<uint32_t *>(m + b_cell);
        out.ent = reinterpret_cast<uint4 *>(m + b_cell + b_fine);
        out.edge = reinterpret_cast<int4 *>(m + b_cell + b_fine + b_ent);
        out.sum = reinterpret_cast<uint16_t *>(m + b_cell + b_fine + b_ent + b_edge);
        out.sb = sb;
        out.n_fine = std::max<uint64_t>(nf, 1);
        out.n_ent = h[0] + h[2] + 4;
        out.n_edge = h[3] + 1;
        if ((e = cudaMemcpy(out.cell, word, size_t(ncell) * 4, cudaMemcpyDeviceToDevice)) != cudaSuccess ||
            (e = cudaMemset(out.fine, 0, 4)) != cudaSuccess ||
            (nf && (e = cudaMemcpy(out.fine, f_word, nf * 4, cudaMemcpyDeviceToDevice)) != cudaSuccess))
            return done(2);
        k_near_coarse<false><<<blocks(ncell), 256>>>(in, cell_off, item_q, item_seg, rad, mask, g, n_ent, n_blk, out.cell,
                                                     out.ent, h[0], tot + 5);
        if (NB)
            k_near_fine<false><<<blocks(nf), 256>>>(in, cell_off, item_q, item_seg, rad, g, sb, blk_cell, nf, f_ent, f_edge,
                                                    h[0], out.fine, out.ent, out.edge, h[2], h[3], tot + 5);
        k_near_sum<<<((1u << (2 * sg)) + 255) / 256, 256>>>(g, sg, out.cell, out.sum, tot + 4, out.ent + (out.n_ent - 4),
                                                            out.edge + h[3]);
        if ((e = cudaGetLastError()) != cudaSuccess ||
            (e = cudaMemcpy(h + 4, tot + 4, 16, cudaMemcpyDeviceToHost)) != cudaSuccess)
            return done(2);
        if (h[5])
            return done(3);
        out.sum_resolved = double(h[4]) / double(uint64_t(1) << (2 * sg));
        return done(0);
    }
}

cudaError_t disk_summary(const uint32_t *cell, int g, uint16_t *sum, unsigned long long *n, double *sum_resolved)
{
    const int sg = std::min(g, kSumLog2);
    unsigned long long h = 0;
    cudaError_t e = cudaMemset(n, 0, 8);
    if (e == cudaSuccess) {
        k_near_sum<<<((1u << (2 * sg)) + 255) / 256, 256>>>(g, sg, cell, sum, n, nullptr, nullptr);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaMemcpy(&h, n, 8, cudaMemcpyDeviceToHost);
    *sum_resolved = double(h) / double(uint64_t(1) << (2 * sg));
    return e;
}

} // namespace spx
