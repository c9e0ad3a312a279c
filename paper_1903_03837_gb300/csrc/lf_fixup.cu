// lf_fixup.cu -- the exact pass over the rays whose neighbour order the render
// or backward kernel left uncertain, one warp per queued ray.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "lf_ray.cuh"

namespace lfk {

// Tap (i, j) of the blend: weight-scaled texel accumulated in FP32 pairs.
template <int DT>
__device__ __forceinline__ void blend_tap(const RenderParamsBase &p, size_t row, int32_t j, float w, bool live,
                                          int32_t j0, float2 &in_xy, float2 &in_zw)
{
    // a dead tap reads column j0 of its row (finite) with weight 0: a branch
    // around the load costs more than the load; j0 is the lane's nearest
    // direction, so in a live row that texel is loaded anyway (an L1 hit)
    const float4 t = texel<DT>(p.texels, LF_DINDEX(row + (uint32_t)(live ? j : j0), (uint64_t)p.rows_valid * p.N,
                                                   p.status, kStatusDebugTexel));
    w = live ? w : 0.0f;
    const float2 w2 = make_float2(w, w);
    in_xy = ffma2(w2, make_float2(t.x, t.y), in_xy);
    in_zw = ffma2(w2, make_float2(t.z, t.w), in_zw);
}

// A set the render kernel settled gives the same samples by its search again
// (in every lane alike); one marked in pend, or any of a ray whose image is
// left to this pass, is ranked by the whole warp.
__device__ __forceinline__ TopK<5> settled_or_ranked(const RenderParamsBase &p, const PointSetK &P, float3 h,
                                                     uint32_t pend, uint32_t bit)
{
    if (pend & (bit | kPendImage)) return coop_knn5(P, p.sphere, h);
    float3 qh, ql;
    unit_hit_df(p.sphere, h, qh, ql);
    bool unc = false;
    const TopK<5> r = knn5(P, qh, ql, candidate_source(P, qh), p.status, unc);
    return unc ? coop_knn5(P, p.sphere, h) : r;          // the same in every lane
}

// One ray rendered (or its gradient scattered) by a whole warp: the sets
// marked in pend ranked exactly by coop_knn5, weights as in the render kernel,
// then lane 0 blends or scatters the taps of nonzero weight. Every lane of the
// warp calls it with the same pixel (pend = 3 when the queue overflowed).
template <int DT, bool BWD>
__device__ __forceinline__ void exact_ray(const RenderParamsBase &p, const ViewK &v, uint32_t px, uint32_t py,
                                          uint32_t pend)
{
    int32_t io[5], jd[5];
    float wo[5], wd[5];
#pragma unroll
    for (int m = 0; m < 5; ++m) {
        io[m] = jd[m] = -1;
        wo[m] = wd[m] = 0.0f;
    }
    float3 ho, hd;
    bool hit = intersect_sphere(p.sphere, v.eye, camera_dir(v, px, py), ho, hd);
    if (hit) {
        const PointSetK Po = point_set(p, 0), Pd = point_set(p, 1);
        const TopK<5> ro0 = settled_or_ranked(p, Po, ho, pend, 1u), rd0 = settled_or_ranked(p, Pd, hd, pend, 2u);
        TopK<5> ro = ro0, rd = rd0;
        hit = set_weights<5>(p, 0, Po.inv_sigma, ro, wo) && set_weights<5>(p, 1, Pd.inv_sigma, rd, wd);
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            io[m] = hit ? ro.i[m] : -1;
            jd[m] = hit ? rd.i[m] : -1;
            wo[m] = hit ? wo[m] : 0.0f;
            wd[m] = hit ? wd[m] : 0.0f;
        }
    }
    if ((threadIdx.x & 31u) != 0u) return;
    if constexpr (BWD) {
        if (!hit) return;
        const float4 g = grad_of(p, v.out_offset + (uint64_t)py * v.width + px);
#pragma unroll
        for (int a = 0; a < 5; ++a) {
            if (wo[a] == 0.0f || (uint32_t)io[a] >= p.rows_valid) continue;
#pragma unroll
            for (int b = 0; b < 5; ++b) {
                if (wd[b] == 0.0f || jd[b] < 0) continue;
                const float W = wo[a] * wd[b];
                add_to_grad(p, (uint64_t)io[a] * p.N + (uint64_t)jd[b], make_float4(W * g.x, W * g.y, W * g.z, W * g.w));
            }
        }
    } else {
        const uint64_t pix = pixel_index(v, px, py);
        if (p.idx) {
            if (p.nearest_only) {
                reinterpret_cast<int2 *>(p.idx)[pix] = make_int2(io[0], jd[0]);
            } else {
                store_idx<5>(p, pix, io, jd);
            }
        }
        if (!(pend & kPendImage)) return;                // the render kernel has stored the image
        float2 acc_xy = make_float2(0.f, 0.f), acc_zw = make_float2(0.f, 0.f);
#pragma unroll
        for (int a = 0; a < 5; ++a) {
            const bool la = wo[a] != 0.0f;
            const int32_t i = la ? io[a] : 0;
            float s = wo[a];
            if constexpr (DT == kF16C4 || DT == kE4M3C4) s *= la ? __ldg(p.scales + i) : 0.0f;
            const size_t row = (size_t)i * p.N;
            float2 in_xy = make_float2(0.f, 0.f), in_zw = make_float2(0.f, 0.f);
#pragma unroll
            for (int b = 0; b < 5; ++b)
                blend_tap<DT>(p, row, jd[b], wd[b], la && wd[b] != 0.0f, max(jd[0], 0), in_xy, in_zw);
            const float2 s2 = make_float2(s, s);
            acc_xy = ffma2(s2, in_xy, acc_xy);
            acc_zw = ffma2(s2, in_zw, acc_zw);
        }
        store_image(p, pix, make_float4(acc_xy.x, acc_xy.y, acc_zw.x, acc_zw.y));
    }
}

// The rays the render kernel queued, one warp per ray; when more were queued
// than the queue holds, every ray of the launch (the exact path gives the same
// result for the rays the render kernel finished). The last CTA to finish
// resets the queue for the next launch (replayable, e.g. from a CUDA graph).
template <int DT, int MAXV, bool BWD>
__global__ void __launch_bounds__(kFixupThreads) fixup_kernel(const __grid_constant__ RenderParams<MAXV> p)
{
    __shared__ uint2 lists[BWD ? kFixupThreads / 32 : 1][BWD ? 2 * kListSlots : 1][32];
    const unsigned long long queued = *reinterpret_cast<volatile unsigned long long *>(p.defer_count);
    const bool all = queued > p.defer_cap;
    const unsigned long long total = all ? p.total_pixels : queued;
    const unsigned long long nw = ((unsigned long long)gridDim.x * blockDim.x) >> 5;
    for (unsigned long long e = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; e < total; e += nw) {
        uint32_t vi = 0, px, py, pend = 3u | (p.nearest_only || p.rows_stored ? kPendImage : 0u);
        if (!all) {
            const unsigned long long it = p.defer_items[e];
            pend = (uint32_t)(it >> 48) & 7u;
            vi = (uint32_t)(it >> 32) & 0xffffu;
            py = (uint32_t)(it >> 16) & 0xffffu;
            px = (uint32_t)it & 0xffffu;
        } else {
            unsigned long long r = e;
            while (r >= (unsigned long long)p.views[vi].width * p.views[vi].height) {
                r -= (unsigned long long)p.views[vi].width * p.views[vi].height;
                ++vi;
            }
            py = (uint32_t)(r / p.views[vi].width);
            px = (uint32_t)(r - (unsigned long long)py * p.views[vi].width);
        }
        if constexpr (BWD) {
            // the backward kernel has scattered the rays it did not queue: the same
            // search (the same bits, in every lane alike) tells them apart
            if (all) {
                const ViewK &v = p.views[vi];
                int co, cd;
                int32_t io[1], jd[1];
                pend = 0;
                if (!certain_miss(v, px, py))
                    ray_lists<0, 32>(p, v, camera_dir(v, px, py), &lists[threadIdx.x >> 5][0][threadIdx.x & 31u], co, cd,
                                     io, jd, pend);
                if (pend == 0) continue;
            }
        }
        exact_ray<DT, BWD>(p, p.views[vi], px, py, pend);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(p.defer_done, 1u) == gridDim.x - 1) {
            atomicExch(p.defer_count, 0ull);
            atomicExch(p.defer_done, 0u);
        }
    }
}

template <int MAXV>
static const void *fixup_fn(int kind, bool bwd)
{
    if (bwd) return (const void *)fixup_kernel<kF32C4, MAXV, true>;
    switch (kind) {
    case kF32C4: return (const void *)fixup_kernel<kF32C4, MAXV, false>;
    case kF32C3: return (const void *)fixup_kernel<kF32C3, MAXV, false>;
    case kF16C4: return (const void *)fixup_kernel<kF16C4, MAXV, false>;
    default: return (const void *)fixup_kernel<kE4M3C4, MAXV, false>;
    }
}

// As many CTAs as the kernel's registers let the SMs hold at once (a few queued
// rays per warp at most), found once per device, kernel and thread.
template <int MAXV>
static cudaError_t launch(int kind, bool bwd, const RenderParams<MAXV> &p, cudaStream_t st)
{
    static thread_local int dev_cached[5] = {-1, -1, -1, -1, -1};
    static thread_local unsigned grids[5];
    const void *f = fixup_fn<MAXV>(kind, bwd);
    const int slot = bwd ? 4 : kind;
    int dev = 0;
    unsigned grid = kFixupCtas;
    if (cudaGetDevice(&dev) == cudaSuccess) {
        if (dev != dev_cached[slot]) {
            int sms = 0, per_sm = 0;
            grids[slot] = kFixupCtas;
            if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, (int)kFixupThreads, 0) == cudaSuccess &&
                sms > 0 && per_sm > 0)
                grids[slot] = (unsigned)(sms * per_sm);
            else
                cudaGetLastError();                      // the default grid serves
            dev_cached[slot] = dev;
        }
        grid = grids[slot];
    }
    void *args[] = {const_cast<RenderParams<MAXV> *>(&p)};
    return launch_kernel(f, dim3(grid), kFixupThreads, args, st);
}

cudaError_t launch_fixup(int kind, bool bwd, const RenderParams<kSmallViews> &p, cudaStream_t st)
{
    return launch(kind, bwd, p, st);
}
cudaError_t launch_fixup(int kind, bool bwd, const RenderParams<kLargeViews> &p, cudaStream_t st)
{
    return launch(kind, bwd, p, st);
}

}  // namespace lfk
