// lf_ray.cuh -- per-ray steps shared by the render, backward and fixup kernels:
// tiles and pixels, the points within the kernel radius of a hit, nearest
// sampling, the texel blend and the image and index stores.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "lf_device.cuh"
#include "lf_kernels.h"

namespace lfk {

// ---------------------------------------------------------------------------
// Tiles
// ---------------------------------------------------------------------------
// Tile t of the launch -> (view, tile column, tile row).
__device__ __forceinline__ void tile_of(const RenderParamsBase &p, const ViewK *views, const uint32_t *prefix,
                                        uint32_t nv, uint32_t t, uint32_t &v, uint32_t &tx, uint32_t &ty)
{
    uint32_t lo = 0, hi = nv;          // largest v with prefix[v] <= t
    while (hi - lo > 1) {
        uint32_t mid = (lo + hi) >> 1;
        if (prefix[mid] <= t) lo = mid; else hi = mid;
    }
    v = lo;
    const uint32_t lt = t - prefix[v], tiles_x = views[v].tiles_x;
    if (p.order == 0) {
        ty = (uint32_t)(((uint64_t)lt * views[v].div_m) >> views[v].div_s);     // lt / tiles_x
        tx = lt - ty * tiles_x;
    } else {                           // strips of kStripTiles tile rows, column by column
        const uint32_t strip = lt / (tiles_x * kStripTiles);
        const uint32_t r = lt - strip * tiles_x * kStripTiles;
        const uint32_t hs = min(kStripTiles, views[v].tiles_y - strip * kStripTiles);
        tx = r / hs;
        ty = strip * kStripTiles + (r - tx * hs);
    }
}

// The CTA's tile: from a grid of (tile columns, tile rows, views) where there is
// one (grid3: raster order, a few views), else by number. False past a smaller
// view's tiles.
template <int MAXV>
__device__ __forceinline__ bool cta_tile(const RenderParams<MAXV> &p, uint32_t &v, uint32_t &tx, uint32_t &ty)
{
    if (MAXV <= kSmallViews && p.grid3) {
        v = blockIdx.z;
        tx = blockIdx.x;
        ty = blockIdx.y;
        return tx < p.views[v].tiles_x && ty < p.views[v].tiles_y;
    }
    tile_of(p, p.views, p.tile_prefix, p.n_views, blockIdx.x, v, tx, ty);
    return true;
}

// Pixel of this thread in tile (tx, ty): tile and warp shapes are powers of
// two, so the mapping is shifts and masks.
__device__ __forceinline__ void pixel_of(const RenderParamsBase &p, uint32_t tx, uint32_t ty, uint32_t &px,
                                         uint32_t &py)
{
    uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t wx_log = p.tw_log - p.ww_log;              // log2(warps per tile row)
    px = (tx << p.tw_log) + ((warp & ((1u << wx_log) - 1u)) << p.ww_log) + (lane & ((1u << p.ww_log) - 1u));
    py = (ty << p.th_log) + ((warp >> wx_log) << (5u - p.ww_log)) + (lane >> p.ww_log);
}

// True when no pixel of tile (tx, ty) can hit S: the tile lies outside the
// view's screen bound of the rays that certain_miss keeps.
__device__ __forceinline__ bool tile_misses(const RenderParamsBase &p, const ViewK &v, uint32_t tx, uint32_t ty)
{
    const uint32_t x0 = tx << p.tw_log, y0 = ty << p.th_log;
    return x0 >= v.sx1 || x0 + p.tile_w <= v.sx0 || y0 >= v.sy1 || y0 + p.tile_h <= v.sy0;
}

__device__ __forceinline__ PointSetK point_set(const RenderParamsBase &p, int s)
{
    PointSetK P;
    P.hi = s ? p.pd.hi : p.po.hi;
    P.lo = s ? p.pd.lo : p.po.lo;
    P.xy = s ? p.pd.xy : p.po.xy;
    P.n = s ? p.pd.n : p.po.n;
    P.nf = s ? p.pd.nf : p.po.nf;
    P.nhalf = s ? p.pd.nhalf : p.po.nhalf;
    P.zpole = s ? p.pd.zpole : p.po.zpole;
    P.inv_sigma = s ? p.pd.inv_sigma : p.po.inv_sigma;
    P.sigma2 = s ? p.pd.sigma2 : p.po.sigma2;
    P.zone0 = s ? p.pd.zone0 : p.po.zone0;
    P.zstep_h = s ? p.pd.zstep_h : p.po.zstep_h;
    P.zstep_l = s ? p.pd.zstep_l : p.po.zstep_l;
    P.z0_h = s ? p.pd.z0_h : p.po.z0_h;
    P.z0_l = s ? p.pd.z0_l : p.po.z0_l;
    P.zstep_c = s ? p.pd.zstep_c : p.po.zstep_c;
    P.zstep_r = s ? p.pd.zstep_r : p.po.zstep_r;
    P.zgrid = s ? p.pd.zgrid : p.po.zgrid;
    return P;
}

// Queues ray (view vi, pixel px, py) for the fixup kernel; bit s of pend marks
// a set whose search was not certain, kPendImage that the image of the ray is
// left to the fixup kernel too. When the queue is full the count still grows
// past defer_cap, which tells the fixup kernel to take every ray.
constexpr uint32_t kPendImage = 4u;
__device__ __forceinline__ void defer_push(const RenderParamsBase &p, uint32_t vi, uint32_t px, uint32_t py,
                                           uint32_t pend)
{
    const unsigned long long slot = atomicAdd(p.defer_count, 1ull);
    if (slot < p.defer_cap)
        p.defer_items[slot] = ((unsigned long long)pend << 48) | ((unsigned long long)vi << 32) |
                              ((unsigned long long)py << 16) | px;
}

// ---------------------------------------------------------------------------
// The neighbours of nonzero weight.
//
// The tent of radius sigma = sqrt(4 pi / n) (the square root of a point's share
// of the sphere) gives weight 0 to every point at sigma or farther, and the
// points nearer than sigma are always 1 to 5 and the nearest lies within 0.78
// sigma (tests/test_kernel_radius.py: the 6th nearest is at least 1.04 sigma
// away for every n, at the poles too). So the weighted neighbours among the 5
// or 9 nearest are exactly the points within sigma, whatever their order: an
// image needs no ranking, no certificate of an order and no exact pass. Away
// from the poles those points lie among 7 corners of the lattice window in the
// quadrant's turned basis (same test; lattice_corner has the other corners):
//   (0,0) (0,1) (1,0) (1,1) (0,-1) (-1,1) (-1,0).
// Ranking 12 corners with a 37-comparator network, the order certificate and
// the double-float distances of the winners cost about 1,250 thread
// instructions per hit ray more than testing 7 distances against sigma.
//
// A ray's two lists (at most kListSlots entries: point index, squared
// distance) wait in shared memory, one column per thread (STRIDE entries from one
// slot to the next).
// ---------------------------------------------------------------------------
constexpr int kListSlots = 5;

// Squared distance of the unit hit to point i (-kPointPad .. n + kPointPad - 1;
// far outside [0, n)), with dz = q_z - z_i at hand.
__device__ __forceinline__ float dist2_xy(const PointSetK &P, int32_t i, float3 qh, float3 ql, float dz,
                                          uint32_t *status)
{
    // a 32-bit byte offset (below 2^29)
    const uint32_t e = LF_DINDEX((uint32_t)(i + kPointPad), P.n + 2 * kPointPad, status, kStatusDebugPoint);
    const float4 a = __ldg(reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(P.xy) + (uint32_t)(e << 4)));
    const float dx = __fadd_rn(__fsub_rn(qh.x, a.x), __fsub_rn(ql.x, a.z));
    const float dy = __fadd_rn(__fsub_rn(qh.y, a.y), __fsub_rn(ql.y, a.w));
    return __fmaf_rn(dx, dx, __fmaf_rn(dy, dy, __fmul_rn(dz, dz)));
}

// Lists the points within sigma of the unit hit qh + ql in `list` (column of
// this thread); their number (1 to 5). Sets of at most 128 points are scanned,
// and within 8 continuous indices of a pole the 28 points nearest it (the 7
// corners hold every point within sigma from 6 indices on, and no point within
// sigma of such a hit has an index of 24 or more; tests/test_kernel_radius.py).
// Corners past either end of the index range read the cache's padding, points
// far from S. With RANK, `src` gets the candidate source of rank5 and `pre` the
// squared distances of its 12 corners.
template <bool RANK, int STRIDE>
__device__ __forceinline__ int points_within(const PointSetK &P, float3 qh, float3 ql, uint2 *list, uint32_t *status,
                                             Source &src, float (&pre)[kWindow])
{
    const int32_t n = (int32_t)P.n;
    uint2 *w = list;
    const uint2 *const end = list + kListSlots * STRIDE;
    if (!(fabsf(qh.z) > P.zpole)) {
        const Corner c = lattice_corner(P, qh);
        if constexpr (RANK) {
            if (!scan_source(P, qh, src)) src = window_of(P, c);
        }
        // never taken: keeps every access within the padded cache whatever the hit's values are
        const int32_t reach = RANK ? 2 * c.reach : c.reach;
        if (c.b - reach < -kPointPad || c.b + reach >= n + kPointPad) return 0;
        const ZOffset zb = z_offset(P, c.b, qh.z, ql.z);
        const float g0 = __int2float_rn(c.G0), g1 = __int2float_rn(c.G1);      // their sums below are exact
        const int32_t b = c.b, ip = b + c.G0, im = b - c.G0;
        const int32_t idx[7] = {b, b + c.G1, ip, ip + c.G1, b - c.G1, im + c.G1, im};
        const float dz[7] = {__fadd_rn(zb.c, zb.r), z_at(P, zb, g1),  z_at(P, zb, g0), z_at(P, zb, g0 + g1),
                             z_at(P, zb, -g1),      z_at(P, zb, g1 - g0), z_at(P, zb, -g0)};
        float d2[7];
#pragma unroll
        for (int j = 0; j < 7; ++j) d2[j] = dist2_xy(P, idx[j], qh, ql, dz[j], status);
#pragma unroll
        for (int j = 0; j < 7; ++j) {
            if (d2[j] < P.sigma2 && (j < kListSlots || w < end)) {
                *w = make_uint2((uint32_t)idx[j], __float_as_uint(d2[j]));
                w += STRIDE;
            }
        }
        if constexpr (RANK) {
            constexpr int kSlot[7] = {5, 9, 6, 10, 1, 8, 4};
#pragma unroll
            for (int j = 0; j < 7; ++j) pre[kSlot[j]] = d2[j];
            const int32_t ix[5] = {im - c.G1, ip - c.G1, ip + c.G0 - c.G1, ip + c.G0, ip + 2 * c.G1};
            const float dzx[5] = {z_at(P, zb, -g0 - g1), z_at(P, zb, g0 - g1), z_at(P, zb, 2.0f * g0 - g1),
                                  z_at(P, zb, 2.0f * g0), z_at(P, zb, g0 + 2.0f * g1)};
            constexpr int kSlotX[5] = {0, 2, 3, 7, 11};      // slot 14 is window candidate 11
#pragma unroll
            for (int j = 0; j < 5; ++j) pre[kSlotX[j]] = dist2_xy(P, ix[j], qh, ql, dzx[j], status);
        }
    } else {
        if constexpr (RANK) scan_source(P, qh, src);
        const int32_t scan_cnt = n > 128 ? 28 : n, scan0 = n > 128 && qh.z < 0.0f ? n - 28 : 0;
#pragma unroll 4
        for (int j = 0; j < scan_cnt; ++j) {
            const int32_t i = scan0 + j;
            const float d2 = dist2_df(P, LF_DINDEX(i, P.n, status, kStatusDebugPoint), qh, ql);
            if (d2 < P.sigma2 && w < end) {
                *w = make_uint2((uint32_t)i, __float_as_uint(d2));
                w += STRIDE;
            }
        }
    }
    return (int)(w - list) / STRIDE;
}

// The indices of the 5 nearest points in (distance, index) order, -1 past the
// set's size; false when the FP32 distances cannot settle the order, which is
// then left to the exact pass. `src`, `pre`: from points_within (corners outside
// the index range are far, and at least five lie inside it). The distances are those of dist2_xy and dist2_df, whose error is below
// e(d2) = 2^-19 sigma d + 2^-21 d2 (z differences off by at most 2^-20 sigma,
// five roundings of the rest); the keys drop the low bits of a distance for the
// slot. One bound, at the 6th key, serves all: with every one of the top 6 keys'
// upper ends below the next key's lower end by more than 2 e and 2^-40 (far
// above any FP64 rounding of the exact distances), the order and the membership
// of the 5 are the exact ones, since every other key is at least the 6th. About
// 0.2% of searches fail this. A first ranking by FP32 high parts alone (one
// third of the arithmetic on 5 of the 12 corners) is certain less often and
// needs a second, divergent one for 3% of the searches: 4% slower.
__device__ __forceinline__ bool rank5(const PointSetK &P, float3 qh, float3 ql, const Source &src, uint32_t *status,
                                      const float (&pre)[kWindow], int32_t (&ix)[5])
{
    constexpr uint32_t kNone = 0xffffffffu;
    const uint32_t mask = (1u << src.bits) - 1u;
    uint32_t k[12];
    if (src.scan_cnt == 0) {
#pragma unroll
        for (int j = 0; j < kWindow; ++j) k[j] = (__float_as_uint(pre[j]) & ~15u) | slot5(j);
        select7_of12(k);
    } else {
        uint32_t s7[7];
#pragma unroll
        for (int m = 0; m < 7; ++m) s7[m] = kNone;
#pragma unroll 1
        for (int j = 0; j < src.scan_cnt; ++j) {
            const int32_t i = src.b0 + j;
            const float d2 = dist2_df(P, LF_DINDEX(i, P.n, status, kStatusDebugPoint), qh, ql);
            insert7(s7, (__float_as_uint(d2) & ~mask) | (uint32_t)j);
        }
#pragma unroll
        for (int m = 0; m < 7; ++m) k[m] = s7[m];
    }
    const float d6 = fminf(__uint_as_float(k[5] | mask), 4.5f);   // an empty slot is all ones: 4.5 > any chord
    const float e = __fmaf_rn(0x1p-21f, d6, 0x1p-19f * sqrt_approx(d6 * P.sigma2));
    const float gap = __fmaf_rn(2.0f, e, 0x1p-40f);
    bool sure = true;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        sure &= (k[m + 1] == kNone) |
                (__fsub_rn(__uint_as_float(k[m + 1] & ~mask), __uint_as_float(k[m] | mask)) > gap);
        ix[m] = k[m] != kNone ? source_index(src, k[m] & mask) : -1;
    }
    return sure;
}

// The list of a scanned set from its ranked indices: the points within sigma are
// among the 5 nearest (even where the order is not certain: the 6th lies beyond
// 1.04 sigma), listed by index as the scan would.
template <int STRIDE, int K>
__device__ __forceinline__ int list_ranked(const PointSetK &P, float3 qh, float3 ql, const int32_t (&ix)[K], uint2 *list)
{
    float d2[kListSlots];
    int c = 0;
#pragma unroll
    for (int m = 0; m < kListSlots; ++m) {
        d2[m] = dist2_df(P, max(ix[m], 0), qh, ql);
        if (ix[m] < 0) d2[m] = 8.0f;
    }
#pragma unroll
    for (int m = 0; m < kListSlots; ++m) {
        if (!(d2[m] < P.sigma2) || ix[m] < 0) continue;
        int at = 0;
#pragma unroll
        for (int k = 0; k < kListSlots; ++k) at += d2[k] < P.sigma2 && ix[k] >= 0 && ix[k] < ix[m] ? 1 : 0;
        list[at * STRIDE] = make_uint2((uint32_t)ix[m], __float_as_uint(d2[m]));
        ++c;
    }
    return c;
}

// Tent weight of a listed point.
__device__ __forceinline__ float tent(float d2, float inv_sigma)
{
    return __saturatef(__fmaf_rn(-sqrt_approx(d2), inv_sigma, 1.0f));
}
// A quarter of it (the same bits, scaled).
__device__ __forceinline__ float quarter_tent(float d2, float inv_sigma)
{
    return __saturatef(__fmaf_rn(-sqrt_approx(d2), 0.25f * inv_sigma, 0.25f));
}

// Nearest sampling: the list becomes its nearest entry, with distance 0 (weight
// 1). The FP32 distances are off by at most 2^-20 sigma per component difference
// in z and 2^-22 of the result otherwise, so by 2^-19 sigma d + 2^-21 d^2; where the
// second is within twice that (and 2^-40) of the first, a few rays of an image, the
// listed points are compared in double-float as the exact pass does. False when
// that cannot tell either. Leaving those few rays to the exact pass kept the device
// for 14 us of its latency behind a 33 us render; now its queue is empty (3 us).
template <int STRIDE>
__device__ __forceinline__ bool nearest_listed(const PointSetK &P, float3 qh, float3 ql, uint2 *list, int c)
{
    float d1 = 8.0f, d2 = 8.0f;
    uint32_t i1 = 0;
#pragma unroll
    for (int m = 0; m < kListSlots; ++m) {
        const uint2 e = list[m * STRIDE];
        const float d = m < c ? __uint_as_float(e.y) : 8.0f;
        i1 = d < d1 ? e.x : i1;
        d2 = fminf(d2, fmaxf(d, d1));
        d1 = fminf(d1, d);
    }
    d2 = fminf(d2, P.sigma2);                            // a second point beyond the list is at sigma or farther
    const float err = __fmaf_rn(0x1p-20f, d2, __fmaf_rn(0x1p-18f, sqrt_approx(d2 * P.sigma2), 0x1p-40f));
    bool sure = d2 - d1 > err;
    if (!sure) {
        df b1{8.0f, 0.0f}, b2{8.0f, 0.0f};
#pragma unroll 1
        for (int m = 0; m < c; ++m) {
            const int32_t i = (int32_t)list[m * STRIDE].x;
            const df d = dist2_dd(P, i, qh, ql);
            if (dd_less(d, i, b1, (int32_t)i1)) {
                b2 = b1;
                b1 = d;
                i1 = (uint32_t)i;
            } else if (d.h < b2.h || (d.h == b2.h && d.l < b2.l)) {
                b2 = d;
            }
        }
        sure = __fadd_rn(__fsub_rn(b2.h, b1.h), __fsub_rn(b2.l, b1.l)) > 2.0f * tier2_err(b2.h);
    }
    list[0] = make_uint2(i1, 0u);
    return sure;
}

// Upper-hemisphere tables: keeps the listed origins whose rows are stored.
template <int STRIDE>
__device__ __forceinline__ int keep_stored(uint2 *list, int c, uint32_t rows)
{
    int k = 0;
#pragma unroll 1
    for (int m = 0; m < c; ++m) {
        const uint2 e = list[m * STRIDE];
        if (e.x < rows) list[STRIDE * k++] = e;
    }
    return k;
}

// Upper-hemisphere tables, a hit with no stored origin within sigma: if the
// nearest stored origin is among the 5 nearest origins it takes weight 1, else
// the ray is masked. Returns the number of listed points (1 or 0); sets
// `uncertain` when the distances are too close to tell (nearest_listed's
// bound, taken at 1.75 sigma, beyond which no 5th nearest lies).
__device__ __forceinline__ int nearest_stored(const PointSetK &P, float3 qh, float3 ql, uint32_t rows, uint2 *list,
                                              bool &uncertain)
{
    const float sigma = sqrtf(P.sigma2);
    // row i is stored iff z_i > 0 (up to the middle row of an odd count, z = 0)
    if (qh.z < -1.75f * sigma) return 0;
    const Source src = candidate_source(P, qh);
    const int total = src.scan_cnt ? src.scan_cnt : kWindow;
    const float err = __fmaf_rn(0x1p-16f, P.sigma2, 0x1p-40f);
    float best = 8.0f;
    int32_t ib = 0;
    for (int pass = 0, nearer = 0;; ++pass) {
        // pass 0: the nearest stored origin; pass 1: how many others are nearer
#pragma unroll 1
        for (int j = 0; j < total; ++j) {
            const int32_t i = source_index(src, src.scan_cnt ? (uint32_t)j : slot5(j));
            if ((uint32_t)i >= P.n) continue;
            const float d2 = dist2_df(P, i, qh, ql);
            if (pass == 0) {
                if ((uint32_t)i < rows && d2 < best) {
                    best = d2;
                    ib = i;
                }
            } else if (i != ib) {
                nearer += d2 < best ? 1 : 0;
                uncertain |= fabsf(d2 - best) <= err;
            }
        }
        if (pass == 0) {
            if (best > 4.5f) return 0;                   // no stored origin in the window
        } else {
            if (nearer >= 5) return 0;
            list[0] = make_uint2((uint32_t)ib, 0u);
            return 1;
        }
    }
}

// Hits and lists of one ray of unit direction d; with IDX (5 or 9) also the
// indices of its nearest points in (distance, index) order. False for a miss or
// a masked ray. Bits of `pend`: defer_push. `lists`: this thread's column of the
// origin list, the direction list after it.
template <int IDX, int STRIDE>
__device__ __forceinline__ bool ray_lists(const RenderParamsBase &p, const ViewK &v, float3 d, uint2 *lists, int &co,
                                          int &cd, int32_t (&io)[IDX ? IDX : 1], int32_t (&jd)[IDX ? IDX : 1],
                                          uint32_t &pend)
{
    __shared__ int s_stash[IDX ? IDX * kMaxBlock : 1];   // the origins' indices during the second search
    float3 ho, hd;
    if (!intersect_sphere(p.sphere, v.eye, d, ho, hd)) return false;
    // Without ranking, a copy of the search for each set: their constants are
    // operands of the instructions (64 uneven views 3.44 -> 3.29 ms); the ranked
    // searches are too long for the instruction cache twice and share one copy.
    constexpr int kSetUnroll = IDX == 0 ? 2 : 1;
#pragma unroll kSetUnroll
    for (int s = 0; s < 2; ++s) {
        const PointSetK P = point_set(p, s);
        uint2 *list = lists + s * kListSlots * STRIDE;
        float3 qh, ql;
        unit_hit_df(p.sphere, s ? hd : ho, qh, ql);
        Source src;
        float pre[kWindow];
        int c = 0;
        // a ranking of a whole set (at most 128 points) has scanned it already: 16% of
        // an index render of 110 directions
        const bool whole = IDX != 0 && P.n <= 128;
        if (whole)
            scan_source(P, qh, src);
        else
            c = points_within<IDX == 5, STRIDE>(P, qh, ql, list, p.status, src, pre);
        int32_t ix[IDX ? IDX : 1];
        if constexpr (IDX == 5) {
            if (!rank5(P, qh, ql, src, p.status, pre, ix)) pend |= 1u << s;
        } else if constexpr (IDX == 9) {
            const TopK<9> r = knn9(P, p.sphere, s ? hd : ho, qh, ql, candidate_source(P, qh), p.status);
#pragma unroll
            for (int m = 0; m < 9; ++m) ix[m] = r.i[m];
        }
        if constexpr (IDX != 0) {
            if (whole) c = list_ranked<STRIDE>(P, qh, ql, ix, list);
        }
        if (p.nearest_only) {
            if (!nearest_listed<STRIDE>(P, qh, ql, list, c)) pend |= (1u << s) | kPendImage;
            c = s == 0 && list[0].x >= p.rows_valid ? 0 : 1;
        } else if (s == 0 && p.rows_stored) {
            c = keep_stored<STRIDE>(list, c, p.rows_stored);
            if (c == 0) {
                // no stored origin within sigma: the nearest stored one of the 5 (9) nearest, if any
                if constexpr (IDX == 9) {
#pragma unroll
                    for (int m = 8; m >= 0; --m)
                        if ((uint32_t)ix[m] < p.rows_stored) {
                            list[0] = make_uint2((uint32_t)ix[m], 0u);
                            c = 1;
                        }
                } else {
                    bool unc = false;
                    c = nearest_stored(P, qh, ql, p.rows_stored, list, unc);
                    if (unc) pend |= 1u | kPendImage;
                }
            }
        }
        if (pend & kPendImage) return true;              // the fixup kernel renders this ray
        if (c == 0) {
            pend = 0;
            return false;
        }
        if (s == 0) {
            co = c;
            if constexpr (IDX != 0) {
#pragma unroll
                for (int m = 0; m < IDX; ++m) s_stash[m * kMaxBlock + threadIdx.x] = ix[m];
            }
        } else {
            cd = c;
            if constexpr (IDX != 0) {
#pragma unroll
                for (int m = 0; m < IDX; ++m) jd[m] = ix[m];
            }
        }
    }
    if constexpr (IDX != 0) {
#pragma unroll
        for (int m = 0; m < IDX; ++m) io[m] = s_stash[m * kMaxBlock + threadIdx.x];
    }
    return true;
}

// ---------------------------------------------------------------------------
// Blend and stores
// ---------------------------------------------------------------------------
// Packed FP32 pair FMA (one instruction for two lanes of a texel).
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c)
{
    unsigned long long ra = *reinterpret_cast<unsigned long long *>(&a);
    unsigned long long rb = *reinterpret_cast<unsigned long long *>(&b);
    unsigned long long rc = *reinterpret_cast<unsigned long long *>(&c);
    unsigned long long rd;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(rd) : "l"(ra), "l"(rb), "l"(rc));
    return *reinterpret_cast<float2 *>(&rd);
}

// binary16 image: the FP32 result rounded once (half the bytes to read back).
__device__ __forceinline__ void store_f16(float *out, uint32_t C, uint64_t pix, float4 acc)
{
    const __half2 xy = __floats2half2_rn(acc.x, acc.y), zw = __floats2half2_rn(acc.z, acc.w);
    if (C == 4) {
        uint2 v;
        v.x = *reinterpret_cast<const uint32_t *>(&xy);
        v.y = *reinterpret_cast<const uint32_t *>(&zw);
        __stcs(reinterpret_cast<uint2 *>(out) + pix, v);
    } else {
        unsigned short *o = reinterpret_cast<unsigned short *>(out) + pix * 3;
        __stcs(o, __half_as_ushort(__low2half(xy)));
        __stcs(o + 1, __half_as_ushort(__high2half(xy)));
        __stcs(o + 2, __half_as_ushort(__low2half(zw)));
    }
}

__device__ __forceinline__ uint64_t pixel_index(const ViewK &v, uint32_t px, uint32_t py)
{
    return v.out_offset + (uint64_t)py * v.width + px;
}

__device__ __forceinline__ void store_image(const RenderParamsBase &p, uint64_t pix, float4 acc)
{
    if (p.out_f16) {
        store_f16(p.out, p.C, pix, acc);
    } else if (p.C == 4) {
        __stcs(reinterpret_cast<float4 *>(p.out) + pix, acc);
    } else {
        float *o = p.out + pix * 3;
        __stcs(o, acc.x);
        __stcs(o + 1, acc.y);
        __stcs(o + 2, acc.z);
    }
}

// The K origin and K direction indices of one ray.
template <int K>
__device__ __forceinline__ void store_idx(const RenderParamsBase &p, uint64_t pix, const int32_t (&io)[K],
                                          const int32_t (&jd)[K])
{
    int2 *q = reinterpret_cast<int2 *>(p.idx + pix * (2 * K));
    int32_t v[2 * K];
#pragma unroll
    for (int m = 0; m < K; ++m) {
        v[m] = io[m];
        v[K + m] = jd[m];
    }
#pragma unroll
    for (int m = 0; m < K; ++m) q[m] = make_int2(v[2 * m], v[2 * m + 1]);
}

// Weights of one set's neighbours r (set 0: origins, 1: directions) by the
// sampling mode; false when the ray is masked (an upper-hemisphere table with
// no stored origin neighbour).
template <int K>
__device__ __forceinline__ bool set_weights(const RenderParamsBase &p, int s, float inv_sigma, TopK<K> &r,
                                            float (&w)[K])
{
    if (p.nearest_only) {
        // nearest sampling: the nearest point alone (Section 2, Fig. 2)
        if (s == 0 && p.rows_stored && (uint32_t)r.i[0] >= p.rows_stored) return false;
#pragma unroll
        for (int m = 0; m < K; ++m) w[m] = m == 0 ? 1.0f : 0.0f;
#pragma unroll
        for (int m = 1; m < K; ++m) r.i[m] = -1;
        return true;
    }
    if (s == 0 && p.rows_stored) return tent_weights_kept(r.d2, r.i, r.cnt, inv_sigma, p.rows_stored, w);
    tent_weights(r.d2, r.cnt, inv_sigma, w);
    return true;
}

__device__ __forceinline__ void add_to_grad(const RenderParamsBase &p, uint64_t key, float4 sum)
{
    key = LF_DINDEX(key, (uint64_t)p.rows_valid * p.N, p.status, kStatusDebugGrad);
    if (p.C == 4) {
        atomicAdd(reinterpret_cast<float4 *>(p.grad) + key, sum);
    } else {
        // 12 bytes: the 8-byte-aligned pair of the three floats, and the third
        float *q = p.grad + key * 3;
        const bool odd = (reinterpret_cast<uintptr_t>(q) & 4u) != 0;
        atomicAdd(reinterpret_cast<float2 *>(q + (odd ? 1 : 0)), odd ? make_float2(sum.y, sum.z) : make_float2(sum.x, sum.y));
        atomicAdd(q + (odd ? 0 : 2), odd ? sum.x : sum.z);
    }
}

// dL/d(image) of pixel pix.
__device__ __forceinline__ float4 grad_of(const RenderParamsBase &p, uint64_t pix)
{
    if (p.C == 4) return __ldg(reinterpret_cast<const float4 *>(p.grad_out) + pix);
    const float *q = p.grad_out + pix * 3;
    return make_float4(__ldg(q), __ldg(q + 1), __ldg(q + 2), 0.f);
}

}  // namespace lfk
