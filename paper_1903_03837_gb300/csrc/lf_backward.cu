// lf_backward.cu -- backward scatter kernels of the light-field sampling path
// (LumiPath, arXiv 1903.03837, Section 2): one thread per camera ray, tiles as
// in the render kernels; grad[i_a][j_b] += W_ab g over the taps of nonzero
// weight.
//
// The rays of a warp (8 x 4 pixels) share most of their neighbours, so a warp
// sums its rays' taps first: the distinct origins (I) and directions (J) of its
// rays are listed, each ray's weights written as a column of an I x 32 and a
// J x 32 matrix in shared memory, and the I x J sums
//   G[a][b] = sum over rays r of wo[a][r] wd[b][r] g[r]
// divided over the lanes, a pair (a, b) at a time: one atomic per texel and warp.
// On the fit of 32 views of 512^2 into a 16,384 x 512 table I is 5 to 8 and J 3
// to 5: 0.35 ms for its 8.4 M rays (68% hit), search included, where 25 taps a ray
// of ballots, shuffles and group sums took 0.93 from the forward's indices and
// more with a search. Issue-bound (73% of the slots, ALU pipe 56%, FMA 32%).
// Warps with more distinct neighbours than kMaxO or kMaxD (small views of large
// tables) sum tap by tap over the lanes that share a texel: a dense matrix would
// hold mostly zeros.
#include <cuda_runtime.h>

#include "lf_ray.cuh"

// Resident CTAs of kMaxBlock threads per SM the register budget is cut for: the
// fit's forward and backward took 631 us at 5 (now 643), 640 at 4, 35 more at 3.
#ifndef LF_MIN_BLOCKS_BWD
#define LF_MIN_BLOCKS_BWD 5
#endif

namespace lfk {

constexpr int kMaxO = 16, kMaxD = 8;     // distinct origins, directions of a warp's matrices
constexpr int kRowF = 36;                // floats per matrix row: 32 rays, rows on different banks
// Shared memory of one warp: the rays' two lists, then (they are in registers by
// then) the matrices, the image gradient of the rays and the neighbours' indices,
// or the neighbours and weights for the tap-by-tap sum.
template <int K>
struct WarpScratch {
    static constexpr int kLists = 2 * kListSlots * 32 * 8, kTaps = 4 * K * 32 * 4;
    static constexpr int kMats = (kMaxO + kMaxD) * kRowF * 4 + 32 * 16 + (kMaxO + kMaxD) * 4;
    static constexpr int kBytes = (kMats > kTaps ? (kMats > kLists ? kMats : kLists) : (kTaps > kLists ? kTaps : kLists));
    __align__(16) unsigned char b[kBytes];
};

// Position of the n-th (0-based) set bit of m (m has more than n set bits).
__device__ __forceinline__ int nth_set_bit(unsigned m, int n)
{
    int pos = 0, c;
    c = __popc(m & 0xffffu); if (n >= c) { n -= c; m >>= 16; pos += 16; }
    c = __popc(m & 0xffu);   if (n >= c) { n -= c; m >>= 8;  pos += 8; }
    c = __popc(m & 0xfu);    if (n >= c) { n -= c; m >>= 4;  pos += 4; }
    c = __popc(m & 0x3u);    if (n >= c) { n -= c; m >>= 2;  pos += 2; }
    c = (int)(m & 1u);       if (n >= c) { pos += 1; }
    return pos;
}

// Sum of `val` over the lanes of this lane's group `grp` (lanes holding the
// same texel key), delivered to the group's lowest lane: a binary tree over the
// members' ranks, log2(largest group) rounds. Every lane of the warp calls it.
__device__ __forceinline__ float4 group_sum_tree(float4 val, unsigned grp, unsigned lane)
{
    const int rank = __popc(grp & ((1u << lane) - 1u));
    const int size = __popc(grp);
    const int maxsize = (int)__reduce_max_sync(0xffffffffu, (unsigned)size);
    for (int off = 1; off < maxsize; off <<= 1) {
        bool recv = (rank & (2 * off - 1)) == 0 && rank + off < size;
        int src = recv ? nth_set_bit(grp, rank + off) : (int)lane;
        float4 o;
        o.x = __shfl_sync(0xffffffffu, val.x, src);
        o.y = __shfl_sync(0xffffffffu, val.y, src);
        o.z = __shfl_sync(0xffffffffu, val.z, src);
        o.w = __shfl_sync(0xffffffffu, val.w, src);
        if (recv) {
            val.x += o.x; val.y += o.y; val.z += o.z; val.w += o.w;
        }
    }
    return val;
}

// The taps of a warp's rays one at a time (every lane of the warp calls it; dead
// entries have weight 0): lanes that hold the same texel are summed first, by a
// butterfly over the warp when all of them do, else by a tree per group, and one
// atomic per group. The loop over origins stays rolled (instruction-cache
// footprint); both sets are read from shared memory (a run-time index into
// registers would move them to local memory).
template <int K>
__device__ __forceinline__ void scatter_taps(const RenderParamsBase &p, int *s, const uint32_t (&io)[K],
                                             const uint32_t (&jd)[K], const float (&wo)[K], const float (&wd)[K],
                                             float4 g)
{
    const unsigned lane = threadIdx.x & 31;
    __syncwarp();
#pragma unroll
    for (int m = 0; m < K; ++m) {
        s[m * 32 + lane] = (int)io[m];
        s[(K + m) * 32 + lane] = __float_as_int(wo[m]);
        s[(2 * K + m) * 32 + lane] = (int)jd[m];
        s[(3 * K + m) * 32 + lane] = __float_as_int(wd[m]);
    }
#pragma unroll 1
    for (int a = 0; a < K; ++a) {
        const uint32_t ia = (uint32_t)s[a * 32 + lane];
        const float wa = __int_as_float(s[(K + a) * 32 + lane]);
        if (!__any_sync(0xffffffffu, wa != 0.0f)) continue;
#pragma unroll
        for (int b = 0; b < K; ++b) {
            const uint32_t jb = (uint32_t)s[(2 * K + b) * 32 + lane];
            const float wb = __int_as_float(s[(3 * K + b) * 32 + lane]);
            const bool live = wa != 0.0f && wb != 0.0f;
            const uint64_t key = live ? (uint64_t)ia * p.N + jb : 0ull;
            const float W = live ? wa * wb : 0.f;
            float4 val = live ? make_float4(W * g.x, W * g.y, W * g.z, W * g.w) : make_float4(0.f, 0.f, 0.f, 0.f);
            const unsigned live_mask = __ballot_sync(0xffffffffu, live);
            if (live_mask == 0u) continue;
            const int leader = __ffs(live_mask) - 1;
            const uint64_t lkey = __shfl_sync(0xffffffffu, key, leader);
            if (__all_sync(0xffffffffu, !live || key == lkey)) {
#pragma unroll
                for (int o = 16; o >= 1; o >>= 1) {
                    val.x += __shfl_xor_sync(0xffffffffu, val.x, o);
                    val.y += __shfl_xor_sync(0xffffffffu, val.y, o);
                    val.z += __shfl_xor_sync(0xffffffffu, val.z, o);
                    val.w += __shfl_xor_sync(0xffffffffu, val.w, o);
                }
                if ((int)lane == leader) add_to_grad(p, lkey, val);
            } else {
                const unsigned grp = __match_any_sync(0xffffffffu, live ? key : ~0ull - lane);
                const float4 sum = group_sum_tree(val, grp, lane);
                if (live && (__ffs(grp) - 1) == (int)lane) add_to_grad(p, key, sum);
            }
        }
    }
}

// The distinct neighbours of a warp's rays: row n of `mat` gets every ray's
// weight of the n-th smallest index, `keys` the index. Returns their number, or
// most + 1 when there are more.
template <int K>
__device__ __forceinline__ int distinct(const uint32_t (&idx)[K], const float (&w)[K], int most, float *mat,
                                        uint32_t *keys)
{
    constexpr uint32_t kNone = 0xffffffffu;
    const unsigned lane = threadIdx.x & 31;
    uint32_t left[K];
#pragma unroll
    for (int m = 0; m < K; ++m) left[m] = w[m] != 0.0f ? idx[m] : kNone;
    for (int n = 0;; ++n) {
        uint32_t least = left[0];
#pragma unroll
        for (int m = 1; m < K; ++m) least = min(least, left[m]);
        const uint32_t key = __reduce_min_sync(0xffffffffu, least);
        if (key == kNone) return n;
        if (n == most) return most + 1;
        float x = 0.0f;
#pragma unroll
        for (int m = 0; m < K; ++m) {
            const bool here = left[m] == key;
            x += here ? w[m] : 0.0f;
            left[m] = here ? kNone : left[m];
        }
        mat[n * kRowF + lane] = x;
        if (lane == 0) keys[n] = key;
    }
}

// The gradient of a warp's rays (every lane of the warp calls it; a ray without
// a hit has weights 0 only).
template <int K>
__device__ __forceinline__ void scatter_warp(const RenderParamsBase &p, WarpScratch<K> &ws, const uint32_t (&io)[K],
                                             const uint32_t (&jd)[K], const float (&wo)[K], const float (&wd)[K],
                                             float4 g)
{
    const unsigned lane = threadIdx.x & 31;
    float *mo = reinterpret_cast<float *>(ws.b), *md = mo + kMaxO * kRowF;
    float4 *sg = reinterpret_cast<float4 *>(md + kMaxD * kRowF);
    uint32_t *ko = reinterpret_cast<uint32_t *>(sg + 32), *kd = ko + kMaxO;
    __syncwarp();
    // a gradient that is not finite must reach its own ray's texels only: 0 times
    // infinity in another texel's sum would spread it
    const bool finite = isfinite(g.x) && isfinite(g.y) && isfinite(g.z) && isfinite(g.w);
    int I = kMaxO + 1, J = kMaxD + 1;
    if (__all_sync(0xffffffffu, finite)) {
        J = distinct<K>(jd, wd, kMaxD, md, kd);
        if (J <= kMaxD) I = distinct<K>(io, wo, kMaxO, mo, ko);
    }
    if (I > kMaxO) {
        scatter_taps<K>(p, reinterpret_cast<int *>(ws.b), io, jd, wo, wd, g);
        return;
    }
    sg[lane] = g;
    __syncwarp();
    const int pairs = I * J;
    const float inv = __fdividef(1.0f, (float)J);
    for (int q0 = 0; q0 < pairs; q0 += 32) {
        const int q = min(q0 + (int)lane, pairs - 1);
        const int a = (int)(((float)q + 0.5f) * inv), b = q - a * J;    // q < 128, J <= 8: far from a rounding
        const float4 *oa = reinterpret_cast<const float4 *>(mo + a * kRowF);
        const float4 *db = reinterpret_cast<const float4 *>(md + b * kRowF);
        float2 xy = make_float2(0.f, 0.f), zw = make_float2(0.f, 0.f);
#pragma unroll 2
        for (int r = 0; r < 8; ++r) {
            const float4 o = oa[r], d = db[r];
            const float W[4] = {o.x * d.x, o.y * d.y, o.z * d.z, o.w * d.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 gr = sg[4 * r + k];
                const float2 w2 = make_float2(W[k], W[k]);
                xy = ffma2(w2, make_float2(gr.x, gr.y), xy);
                zw = ffma2(w2, make_float2(gr.z, gr.w), zw);
            }
        }
        // texels no ray of the warp touches (and sums of exactly 0) take no atomic
        const bool some = xy.x != 0.0f || xy.y != 0.0f || zw.x != 0.0f || zw.y != 0.0f;
        if (q0 + (int)lane < pairs && some)
            add_to_grad(p, (uint64_t)ko[a] * p.N + kd[b], make_float4(xy.x, xy.y, zw.x, zw.y));
    }
}

// Neighbours and weights of one ray from the indices a forward pass wrote for it
// (idx_in: [P][2K], or [P][2] with nearest sampling): the hits and unit hits are
// recomputed and the weights formed from the distances of these indices. An
// index out of range counts as missing and sets bit 0 of the status word; a ray
// the indices call a hit but that misses S sets bit 1.
template <int K>
__device__ __forceinline__ bool samples_from_idx(const RenderParamsBase &p, const ViewK &v, uint32_t px, uint32_t py,
                                                 uint64_t pix, uint32_t (&io)[K], uint32_t (&jd)[K], float (&wo)[K],
                                                 float (&wd)[K])
{
    const int32_t *q = p.idx_in + pix * (uint64_t)(p.nearest_only ? 2 : 2 * K);
    int32_t ix[2][K];
#pragma unroll
    for (int m = 0; m < K; ++m) ix[0][m] = ix[1][m] = -1;
    if (p.nearest_only) {
        ix[0][0] = __ldg(q);
        ix[1][0] = __ldg(q + 1);
    } else {
#pragma unroll
        for (int m = 0; m < K; ++m) {
            ix[0][m] = __ldg(q + m);
            ix[1][m] = __ldg(q + K + m);
        }
    }
    if (ix[0][0] < 0) return false;
    float3 ho, hd;
    if (!intersect_sphere(p.sphere, v.eye, camera_dir(v, px, py), ho, hd)) {
        atomicOr(p.status, kStatusIdxInput);
        return false;
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const PointSetK P = point_set(p, s);
        const uint32_t stored = s ? P.n : p.rows_valid;
        uint32_t (&id)[K] = s ? jd : io;
        float(&w)[K] = s ? wd : wo;
        float3 qh, ql;
        unit_hit_df(p.sphere, s ? hd : ho, qh, ql);
        float sum = 0.0f;
        int first = -1;
#pragma unroll
        for (int m = K - 1; m >= 0; --m) {
            const bool in = (uint32_t)ix[s][m] < P.n;
            if (!in && ix[s][m] >= 0) atomicOr(p.status, kStatusIndex);
            const bool ok = in && (uint32_t)ix[s][m] < stored;
            const float d2 = dist2_df(P, in ? ix[s][m] : 0, qh, ql);
            id[m] = ok ? (uint32_t)ix[s][m] : 0u;
            w[m] = ok ? (p.nearest_only ? 1.0f : tent(d2, P.inv_sigma)) : 0.0f;
            first = ok ? m : first;
            sum += w[m];
        }
        if (first < 0) return false;
        // all kept neighbours beyond the kernel radius: the first takes weight 1
        const float r = sum > 0.0f ? rcp_approx(sum) : 0.0f;
#pragma unroll
        for (int m = 0; m < K; ++m) w[m] = sum > 0.0f ? w[m] * r : m == first ? 1.0f : 0.0f;
    }
    return true;
}

// SEARCH: the neighbours are searched (0: the points within the kernel radius;
// 9: an upper-hemisphere table with nine neighbours, whose masked rays need the 9
// nearest); otherwise (-1) they come from the forward's indices.
template <int SEARCH, int K>
__device__ __forceinline__ void backward_ray(const RenderParamsBase &p, const ViewK &v, uint32_t vi, bool active,
                                             uint32_t px, uint32_t py, WarpScratch<K> &ws)
{
    uint32_t io[K], jd[K];
    float wo[K], wd[K];
    bool hit = false;
    const uint64_t pix = pixel_index(v, px, py);
    if constexpr (SEARCH < 0) {
        hit = active && samples_from_idx<K>(p, v, px, py, pix, io, jd, wo, wd);
    } else {
        static_assert(K == kListSlots, "a list's slots");
        constexpr int KI = SEARCH ? SEARCH : 1;
        int32_t ni[KI], nj[KI];
        int co = 0, cd = 0;
        uint32_t pend = 0;
        uint2 *lists = reinterpret_cast<uint2 *>(ws.b) + (threadIdx.x & 31);
        hit = active && !certain_miss(v, px, py) &&
              ray_lists<SEARCH, 32>(p, v, camera_dir(v, px, py), lists, co, cd, ni, nj, pend);
        if (pend) {
            defer_push(p, vi, px, py, pend);   // scattered by the fixup kernel
            hit = false;
        }
        if (hit) {
            float so = 0.0f, sd = 0.0f;
#pragma unroll
            for (int m = 0; m < K; ++m) {
                const uint2 e = lists[m * 32], f = lists[(kListSlots + m) * 32];
                io[m] = e.x;
                jd[m] = f.x;
                wo[m] = m < co ? tent(__uint_as_float(e.y), p.po.inv_sigma) : 0.0f;
                wd[m] = m < cd ? tent(__uint_as_float(f.y), p.pd.inv_sigma) : 0.0f;
                so += wo[m];
                sd += wd[m];
            }
            const float r = rcp_approx(so * sd);
#pragma unroll
            for (int m = 0; m < K; ++m) wo[m] *= r;
        }
    }
    if (!__any_sync(0xffffffffu, hit)) return;
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
    if (hit) {
        g = grad_of(p, pix);
    } else {
#pragma unroll
        for (int m = 0; m < K; ++m) {
            io[m] = jd[m] = 0;
            wo[m] = wd[m] = 0.0f;
        }
    }
    scatter_warp<K>(p, ws, io, jd, wo, wd, g);
}

template <int MAXV, int SEARCH, int K>
__global__ void __launch_bounds__(kMaxBlock, K == 5 && SEARCH != 9 ? LF_MIN_BLOCKS_BWD : 2)
    backward_kernel(const __grid_constant__ RenderParams<MAXV> p)
{
    __shared__ WarpScratch<K> ws[kMaxBlock / 32];
    uint32_t v, tx, ty, px, py;
    if (!cta_tile(p, v, tx, ty)) return;
    const ViewK &vw = p.views[v];
    if (SEARCH >= 0 && tile_misses(p, vw, tx, ty)) return;   // given indices are checked against every ray
    pixel_of(p, tx, ty, px, py);
    backward_ray<SEARCH, K>(p, vw, v, px < vw.width && py < vw.height, px, py, ws[threadIdx.x >> 5]);
}

template <int MAXV>
static const void *backward_fn(const RenderParamsBase &p)
{
    if (p.idx_in)
        return p.nine ? (const void *)backward_kernel<MAXV, -1, 9> : (const void *)backward_kernel<MAXV, -1, 5>;
    return p.nine && p.rows_stored ? (const void *)backward_kernel<MAXV, 9, 5>
                                   : (const void *)backward_kernel<MAXV, 0, 5>;
}

template <int MAXV>
static cudaError_t launch(const RenderParams<MAXV> &p, dim3 grid, unsigned block, cudaStream_t st)
{
    void *args[] = {const_cast<RenderParams<MAXV> *>(&p)};
    cudaError_t e = launch_kernel(backward_fn<MAXV>(p), grid, block, args, st);
    // nearest sampling may leave near-ties to the exact pass, an upper-hemisphere table rays at the rim of its rows
    if (e == cudaSuccess && !p.nine && !p.idx_in && (p.nearest_only || p.rows_stored)) e = launch_fixup(kF32C4, true, p, st);
    return e;
}

cudaError_t launch_backward(const RenderParams<kSmallViews> &p, dim3 grid, unsigned block, cudaStream_t st)
{
    return launch(p, grid, block, st);
}
cudaError_t launch_backward(const RenderParams<kLargeViews> &p, dim3 grid, unsigned block, cudaStream_t st)
{
    return launch(p, grid, block, st);
}

}  // namespace lfk
