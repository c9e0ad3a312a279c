// lf_backward.cu -- backward scatter kernel of the light-field sampling path
// (LumiPath, arXiv 1903.03837, Section 2): one thread per camera ray, tiles as
// in the render kernels.
#include <cuda_runtime.h>

#include "lf_ray.cuh"

// Resident CTAs of kMaxBlock threads per SM the register budget is cut for:
// 4 -> 64 registers, 32 warps per SM.
#ifndef LF_MIN_BLOCKS_BWD
#define LF_MIN_BLOCKS_BWD 4
#endif

namespace lfk {

// Indices and normalised weights of one ray of unit direction d (K = 5 or 9
// neighbours per hit); false for a miss. With five neighbours, a set whose tier-1 order was not
// certain sets bit s of `pend` and leaves its samples empty; resolve_pending
// fills them in once the warp has reconverged.
template <int K>
__device__ __forceinline__ bool ray_samples(const RenderParamsBase &p, const ViewK &v, float3 d,
                                            int32_t (&io)[K], int32_t (&jd)[K], float (&wo)[K],
                                            float (&wd)[K], uint32_t &pend)
{
    // The origin set's indices and weights wait in shared memory (one slot per
    // thread, no synchronisation) while the direction set is searched: 2K
    // fewer live registers across the second search.
    __shared__ int s_stash[2 * K * kMaxBlock];
    float3 ho, hd;
    if (!intersect_sphere(p.sphere, v.eye, d, ho, hd)) return false;
    // One copy of the index step serves both sets (instruction-cache footprint).
#pragma unroll 1
    for (int s = 0; s < 2; ++s) {
        const PointSetK P = point_set(p, s);
        TopK<K> r;
        bool unc = false;
            float3 qh, ql;
        unit_hit_df(p.sphere, s ? hd : ho, qh, ql);
        const Source src = candidate_source(P, qh);
        if constexpr (K == 9)
            r = knn9(P, p.sphere, s ? hd : ho, qh, ql, src, p.status);
        else
            r = knn5(P, qh, ql, src, p.status, unc);
        float w[K];
        if (unc) {
            pend |= 1u << s;
#pragma unroll
            for (int m = 0; m < K; ++m) w[m] = 0.0f;
        } else if (!set_weights<K>(p, s, P.inv_sigma, r, w)) {
            pend = 0;
            return false;
        }
        if (s == 0) {
#pragma unroll
            for (int m = 0; m < K; ++m) {
                s_stash[m * kMaxBlock + threadIdx.x] = r.i[m];
                s_stash[(K + m) * kMaxBlock + threadIdx.x] = __float_as_int(w[m]);
            }
        } else {
#pragma unroll
            for (int m = 0; m < K; ++m) {
                jd[m] = r.i[m];
                wd[m] = w[m];
            }
        }
    }
#pragma unroll
    for (int m = 0; m < K; ++m) {
        io[m] = s_stash[m * kMaxBlock + threadIdx.x];
        wo[m] = __int_as_float(s_stash[(K + m) * kMaxBlock + threadIdx.x]);
    }
    return true;
}

// The samples of one ray from the indices a forward pass wrote for it (idx_in:
// [P][2K], or [P][2] with nearest sampling): the hits and unit hits are
// recomputed and the weights formed from the double-float distances of these
// indices -- the same distances, by the same function, as the index step's, so
// the weights are identical. An index out of range counts as missing and sets
// bit 0 of the status word; a ray the indices call a hit but that misses S sets
// bit 1.
template <int K>
__device__ __forceinline__ bool samples_from_idx(const RenderParamsBase &p, const ViewK &v, uint32_t px,
                                                 uint32_t py, uint64_t pix, int32_t (&io)[K], int32_t (&jd)[K],
                                                 float (&wo)[K], float (&wd)[K])
{
    const int32_t *q = p.idx_in + pix * (uint64_t)(p.nearest_only ? 2 : 2 * K);
#pragma unroll
    for (int m = 0; m < K; ++m) io[m] = jd[m] = -1;
    if (p.nearest_only) {
        io[0] = __ldg(q);
        jd[0] = __ldg(q + 1);
    } else {
#pragma unroll
        for (int m = 0; m < K; ++m) {
            io[m] = __ldg(q + m);
            jd[m] = __ldg(q + K + m);
        }
    }
    if (io[0] < 0) return false;
    float3 d = camera_dir(v, px, py);
    float3 ho, hd;
    if (!intersect_sphere(p.sphere, v.eye, d, ho, hd)) {
        atomicOr(p.status, kStatusIdxInput);
        return false;
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        PointSetK P;
        P.hi = s ? p.pd.hi : p.po.hi;
        P.lo = s ? p.pd.lo : p.po.lo;
        P.n = s ? p.pd.n : p.po.n;
        P.inv_sigma = s ? p.pd.inv_sigma : p.po.inv_sigma;
        int32_t (&ix)[K] = s ? jd : io;
        float(&w)[K] = s ? wd : wo;
        float3 qh, ql;
        unit_hit_df(p.sphere, s ? hd : ho, qh, ql);
        float d2[K];
        int cnt = 0;
#pragma unroll
        for (int m = 0; m < K; ++m) {
            const bool ok = (uint32_t)ix[m] < P.n;
            if (!ok && ix[m] >= 0) {
                atomicOr(p.status, kStatusIndex);
                ix[m] = -1;
            }
            d2[m] = ok ? dist2_df(P, ok ? ix[m] : 0, qh, ql) : 0.0f;
            cnt += ok ? 1 : 0;
        }
        if (p.nearest_only) {
#pragma unroll
            for (int m = 0; m < K; ++m) w[m] = m == 0 ? 1.0f : 0.0f;
        } else if (s == 0 && p.rows_stored) {
            if (!tent_weights_kept(d2, ix, cnt, P.inv_sigma, p.rows_stored, w)) return false;
        } else {
            tent_weights(d2, cnt, P.inv_sigma, w);
        }
    }
    return true;
}

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

// The warp-aggregated scatter of the taps of one warp's rays (every lane of
// the warp calls it; lanes without a hit contribute nothing).
template <int K>
__device__ __forceinline__ void backward_taps(const RenderParamsBase &p, bool hit, const int32_t (&io)[K],
                                              const int32_t (&jd)[K], const float (&wo)[K], const float (&wd)[K],
                                              float4 g)
{
    const unsigned lane = threadIdx.x & 31;
    // Both neighbour sets wait in a per-thread shared-memory slot during the tap
    // loop (no synchronisation: each thread reads only its own slot): twenty
    // registers fewer than keeping them live, 8% faster.
    __shared__ int s_bw[4 * K * kMaxBlock];
#pragma unroll
    for (int m = 0; m < K; ++m) {
        s_bw[m * kMaxBlock + threadIdx.x] = io[m];
        s_bw[(K + m) * kMaxBlock + threadIdx.x] = __float_as_int(wo[m]);
        s_bw[(2 * K + m) * kMaxBlock + threadIdx.x] = jd[m];
        s_bw[(3 * K + m) * kMaxBlock + threadIdx.x] = __float_as_int(wd[m]);
    }
#pragma unroll 1
    for (int a = 0; a < K; ++a) {
        const int32_t ia = s_bw[a * kMaxBlock + threadIdx.x];
        const float wa = __int_as_float(s_bw[(K + a) * kMaxBlock + threadIdx.x]);
#pragma unroll
        for (int b = 0; b < K; ++b) {
            const int32_t jb = s_bw[(2 * K + b) * kMaxBlock + threadIdx.x];
            const float wb = __int_as_float(s_bw[(3 * K + b) * kMaxBlock + threadIdx.x]);
            // a tap of weight 0 (beyond the kernel radius in either set) would add
            // exactly 0: it takes no atomic
            bool live = hit && (uint32_t)ia < p.rows_valid && jb >= 0 && wa != 0.0f && wb != 0.0f;
            uint64_t key = live ? (uint64_t)ia * p.N + (uint64_t)jb : 0ull;
            float W = live ? wa * wb : 0.f;
            float4 val = make_float4(W * g.x, W * g.y, W * g.z, W * g.w);
            unsigned live_mask = __ballot_sync(0xffffffffu, live);
            if (live_mask == 0u) continue;
            const int leader = __ffs(live_mask) - 1;
            uint64_t lkey = __shfl_sync(0xffffffffu, key, leader);
            if (__all_sync(0xffffffffu, !live || key == lkey)) {
#pragma unroll
                for (int s = 16; s >= 1; s >>= 1) {
                    val.x += __shfl_xor_sync(0xffffffffu, val.x, s);
                    val.y += __shfl_xor_sync(0xffffffffu, val.y, s);
                    val.z += __shfl_xor_sync(0xffffffffu, val.z, s);
                    val.w += __shfl_xor_sync(0xffffffffu, val.w, s);
                }
                if ((int)lane == leader) add_to_grad(p, lkey, val);
            } else {
                unsigned grp = __match_any_sync(0xffffffffu, live ? key : ~0ull - lane);
                float4 sum = group_sum_tree(val, grp, lane);
                if (live && (__ffs(grp) - 1) == (int)lane) add_to_grad(p, key, sum);
            }
        }
    }
}
// Backward of one ray: grad[i_a][j_b] += W_ab * g for the K x K taps. Lanes that
// hold the same texel key are summed first (warp aggregation): when every live
// lane of the warp has the same key, a butterfly over the warp and one atomic;
// otherwise __match_any_sync groups and a tree sum per group, one atomic per
// group. The loop over origin neighbours stays rolled (instruction-cache
// footprint) and the K direction taps inside it unrolled; both read the
// neighbours from shared memory (a run-time index into register arrays would
// move them to local memory).
template <int K>
__device__ __forceinline__ void backward_ray(const RenderParamsBase &p, const ViewK *v, uint32_t vi, bool active,
                                             uint32_t px, uint32_t py)
{
    int32_t io[K], jd[K];
    float wo[K], wd[K];
#pragma unroll
    for (int m = 0; m < K; ++m) {
        io[m] = jd[m] = -1;
        wo[m] = wd[m] = 0.0f;
    }
    bool hit = false;
    uint32_t pend = 0;
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
    if (active) {
        uint64_t pix = v->out_offset + (uint64_t)py * v->width + px;
        hit = p.idx_in ? samples_from_idx<K>(p, *v, px, py, pix, io, jd, wo, wd)
                       : (!certain_miss(*v, px, py) &&
                          ray_samples<K>(p, *v, camera_dir(*v, px, py), io, jd, wo, wd, pend));
        g = grad_of(p, pix);
    }
    if (pend) {
        defer_push(p, vi, px, py, pend);   // scattered by the fixup kernel
        hit = false;
    }
    if (__any_sync(0xffffffffu, hit)) backward_taps<K>(p, hit, io, jd, wo, wd, g);
}

template <int MAXV, int K>
__global__ void __launch_bounds__(kMaxBlock, K == 5 ? LF_MIN_BLOCKS_BWD : 2)
    backward_kernel(const __grid_constant__ RenderParams<MAXV> p)
{
    uint32_t v, tx, ty, px, py;
    tile_of(p, p.views, p.tile_prefix, p.n_views, blockIdx.x, v, tx, ty);
    const ViewK &vw = p.views[v];
    pixel_of(p, tx, ty, px, py);
    backward_ray<K>(p, &vw, v, px < vw.width && py < vw.height, px, py);
}

template <int MAXV>
static const void *backward_fn(const RenderParamsBase &p)
{
    return p.nine ? (const void *)backward_kernel<MAXV, 9> : (const void *)backward_kernel<MAXV, 5>;
}

template <int MAXV>
static cudaError_t launch(const RenderParams<MAXV> &p, unsigned grid, unsigned block, cudaStream_t st)
{
    void *args[] = {const_cast<RenderParams<MAXV> *>(&p)};
    cudaError_t e = cudaLaunchKernel(backward_fn<MAXV>(p), dim3(grid), dim3(block), args, 0, st);
    // a search may leave near-ties to the exact pass (never with nine neighbours or given indices)
    if (e == cudaSuccess && !p.nine && !p.idx_in) e = launch_fixup(kF32C4, true, p, st);
    return e;
}

cudaError_t launch_backward(const RenderParams<kSmallViews> &p, unsigned grid, unsigned block, cudaStream_t st)
{
    return launch(p, grid, block, st);
}
cudaError_t launch_backward(const RenderParams<kLargeViews> &p, unsigned grid, unsigned block, cudaStream_t st)
{
    return launch(p, grid, block, st);
}

}  // namespace lfk
