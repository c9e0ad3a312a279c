// lf_precompute.cu -- the light-field precompute of Section 2: every ray
// r_k = (O + R p^o_i) + t d_ij of the two SF point sets, with its origin
// jittered on the disk of area A_S / M tangent to S, traced through an
// analytic emission-absorption volume of Gaussian blobs; L^(i,j) is the mean
// over the jittered samples.
//
// One thread per texel, FP32. Per sample the blobs are re-expressed along the
// ray: with f_b = o - mu_b and a_b^2 = log2(e) / (2 s_b^2), the density of blob
// b at step k (t_k = (k + 1/2) dt) is
//   exp2(la_b - y_k^2),  la_b = log2(kappa_b) - a_b^2 |f_b x d|^2,
//                        y_k  = a_b (f_b . d + 1/2 dt) + k (a_b dt),
// two fma and one ex2 per blob-step (blobs in pairs: two packed fma and two ex2 a
// pair, the exponent as y_k^2 - la_b with its sign flipped on the way into ex2).
// The cross product keeps the distance of
// the ray from a narrow blob's centre accurate (|f|^2 - (f.d)^2 would cancel).
// The emission is accumulated per blob, G_b += w_k g_bk with w_k the step's
// compositing weight, and turned into colour once per sample: sum_b G_b emit_b
// (the same sum as sum_k w_k sum_b g_bk emit_b, one fma per blob-step instead
// of three).
#include <cuda_runtime.h>
#include <math.h>

#include "lf_device.cuh"
#include "lf_df.cuh"
#include "lf_kernels.h"

namespace lfk {

constexpr float kLog2e = 1.4426950408889634f;

// 2^x by the hardware approximation (relative error below 2^-22; results
// below 2^-126 flush to zero, far below any contribution that matters here).
__device__ __forceinline__ float ex2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Packed FP32 pairs (one instruction for two blobs).
__device__ __forceinline__ unsigned long long pk(float2 a) { return *reinterpret_cast<unsigned long long *>(&a); }
__device__ __forceinline__ float2 upk(unsigned long long r) { return *reinterpret_cast<float2 *>(&r); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)), "l"(pk(c)));
    return upk(d);
}
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(pk(a)), "l"(pk(b)));
    return upk(d);
}

// (1 - exp(-x)) / x = 1 + x P(x) on [0, 1], P of degree 5 by interpolation at the
// Chebyshev nodes (fit_step_weight.py writes the coefficients: within 4e-8 of it in
// exact arithmetic, 1e-7 in float32). With
// T e^-x = T - w x it takes the place of the exponential of a step's optical depth:
// without that one's error, which the transmittance multiplied up, the table is
// within 1.3e-7 (relative norm) of 64 bits instead of 6 to 8e-7. It spares no XU
// instruction: the dense step's ex2 and reciprocal (past x = 1) are issued in every
// step, 10.1 of them a step for 8 blobs, 50.7 instructions in all (51.7 before).
__device__ __forceinline__ float one_minus_exp_over_x(float x)
{
    float h = 0.00013742418377660215f;
    h = fmaf(h, x, -0.0013248180039227009f);
    h = fmaf(h, x, 0.00830117054283619f);
    h = fmaf(h, x, -0.04165925458073616f);
    h = fmaf(h, x, 0.16666603088378906f);
    h = fmaf(h, x, -0.5f);
    return fmaf(h, x, 1.0f);
}

// CTAs of 256 threads per SM the register budget is cut for (the direct render of 9
// blobs or more: 2), and the unroll of the step loop. Precompute of 16,384 x 512 texels,
// 8 blobs, 4 samples of 64 steps: 3.73 ms at 2 and 2, 3.75 to 3.82 at 3 or 4 CTAs
// or unrolled by 1 or 4. Direct render of 8 views of 512^2: 133 us at 3 and 4, 1
// to 4% more elsewhere. Scalar instead of packed FP32 costs the precompute 10% and
// more.
constexpr int kPreBlocks = 2, kPreUnroll = 2, kVolBlocks = 3, kVolUnroll = 4;

// Radiance collected along o + t d, t in [0, t_end], by the midpoint rule with
// p.steps steps of constant density and emission (see the top of the file):
// (RGB including the background seen through the final transmittance T, and
// 1 - T). BP: pairs of blobs.
template <int BP, int UNROLL>
__device__ __forceinline__ float4 march(const PrecomputeParams &p, float ox, float oy, float oz, float dx,
                                        float dy, float dz, float t_end)
{
    const float dt = t_end / (float)p.steps;
    // per-blob constants of this ray, in pairs: y0, dy and -(la + log2 dt): the step
    // length is folded into the densities, g' = g dt = 2^(la + log2 dt - y^2), so the
    // step's optical depth is sum g' and its weight T (1 - e^-x) / x
    float2 Y0[BP], DY[BP], NL[BP], G2[BP];
    const float l2dt = __log2f(dt);
#pragma unroll
    for (int q = 0; q < BP; ++q) {
        float y0[2], dy0[2], nl[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = 2 * q + h;
            const float4 bp = p.blob_pos[k];
            const float a = p.blob_col[k].w;
            const float fx = ox - bp.x, fy = oy - bp.y, fz = oz - bp.z;
            const float along = fmaf(fx, dx, fmaf(fy, dy, fz * dz));
            const float cx = fy * dz - fz * dy, cy = fz * dx - fx * dz, cz = fx * dy - fy * dx;
            const float perp = fmaf(cx, cx, fmaf(cy, cy, cz * cz));
            y0[h] = a * fmaf(0.5f, dt, along);
            dy0[h] = a * dt;
            nl[h] = k < (int)p.nb ? -(fmaf(-a * a, perp, bp.w) + l2dt) : INFINITY;
        }
        Y0[q] = make_float2(y0[0], y0[1]);
        DY[q] = make_float2(dy0[0], dy0[1]);
        NL[q] = make_float2(nl[0], nl[1]);
        G2[q] = make_float2(0.0f, 0.0f);
    }

    float T = 1.0f;
    if (dt > 0.0f) {
        float kf = 0.0f;
#pragma unroll UNROLL
        for (uint32_t st = 0; st < p.steps; ++st, kf += 1.0f) {
            const float2 kf2 = make_float2(kf, kf);
            float2 g2[BP], sig2;
#pragma unroll
            for (int q = 0; q < BP; ++q) {
                const float2 y = fma2(kf2, DY[q], Y0[q]);
                const float2 n = fma2(y, y, NL[q]);
                g2[q] = make_float2(ex2_approx(-n.x), ex2_approx(-n.y));
                sig2 = q ? add2(sig2, g2[q]) : g2[0];
            }
            // step of constant density: x = sigma dt, weight w = T (1 - e^-x) / x per g',
            // and T e^-x = T - w x
            const float x = sig2.x + sig2.y;
            float w = T * one_minus_exp_over_x(x), Tn = fmaf(-w, x, T);
            if (x > 1.0f) {                              // a dense step, past the polynomial
                const float E = ex2_approx(-x * kLog2e);
                w = T * ((1.0f - E) * rcp_approx(x));
                Tn = T * E;
            }
            T = Tn;
            const float2 w2 = make_float2(w, w);
#pragma unroll
            for (int q = 0; q < BP; ++q) G2[q] = fma2(w2, g2[q], G2[q]);
        }
    }
    float L0 = 0.0f, L1 = 0.0f, L2 = 0.0f;
#pragma unroll
    for (int k = 0; k < 2 * BP; ++k) {
        const float4 bc = p.blob_col[k];
        const float G = k & 1 ? G2[k >> 1].y : G2[k >> 1].x;
        L0 = fmaf(G, bc.x, L0);
        L1 = fmaf(G, bc.y, L1);
        L2 = fmaf(G, bc.z, L2);
    }
    const float bgw = 0.5f * (1.0f + dz);
    return make_float4(fmaf(T, fmaf(p.bg1[0], bgw, p.bg0[0]), L0), fmaf(T, fmaf(p.bg1[1], bgw, p.bg0[1]), L1),
                       fmaf(T, fmaf(p.bg1[2], bgw, p.bg0[2]), L2), 1.0f - T);
}

template <int BP>
__global__ void __launch_bounds__(256, kPreBlocks)
    precompute_kernel(const __grid_constant__ PrecomputeParams p)
{
    const uint64_t total = (uint64_t)p.rows * p.N;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += stride) {
        const uint32_t i = (uint32_t)(t / p.N);
        const uint32_t j = (uint32_t)(t - (uint64_t)i * p.N);
        const float4 ph = __ldg(p.po_hi + i), pl = __ldg(p.po_lo + i);
        const float4 qh = __ldg(p.pd_hi + j), ql = __ldg(p.pd_lo + j);
        const float px = ph.x + pl.x, py = ph.y + pl.y, pz = ph.z + pl.z;

        // chord direction d_ij from the hi/lo parts (-p if the points coincide)
        float dx = (qh.x - ph.x) + (ql.x - pl.x);
        float dy = (qh.y - ph.y) + (ql.y - pl.y);
        float dz = (qh.z - ph.z) + (ql.z - pl.z);
        const float l2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        if (l2 < 1e-24f) {
            dx = -px; dy = -py; dz = -pz;
        } else {
            const float il = rsqrtf(l2);
            dx *= il; dy *= il; dz *= il;
        }

        // unit tangents of S at p along azimuth and polar angle
        const float rho2 = fmaf(px, px, py * py);
        const float irho = rsqrtf(rho2);
        const float ephx = -py * irho, ephy = px * irho;
        const float ethx = px * pz * irho, ethy = py * pz * irho, ethz = -rho2 * irho;
        const float pd = fmaf(px, dx, fmaf(py, dy, pz * dz));    // p . d

        float acc0 = 0.0f, acc1 = 0.0f, acc2 = 0.0f, acc3 = 0.0f;
        for (uint32_t s = 0; s < p.spp; ++s) {
            // origin o = O + R p + off, off in the tangent plane (|off| <= disk_r)
            float offx = 0.0f, offy = 0.0f, offz = 0.0f;
            if (p.jitter) {
                const uint64_t ctr = 2ull * (((uint64_t)i * p.N + j) * p.spp + s);
                const float u1 = (float)(uint32_t)(splitmix64(p.seed, ctr) >> 40) * 0x1p-24f;
                const float u2 = (float)(uint32_t)(splitmix64(p.seed, ctr + 1) >> 40) * 0x1p-24f;
                const float r = p.disk_r * sqrtf(u1);
                float sa, ca;
                sincospif(2.0f * u2, &sa, &ca);
                offx = r * fmaf(ca, ephx, sa * ethx);
                offy = r * fmaf(ca, ephy, sa * ethy);
                offz = r * (sa * ethz);
            }
            const float ox = fmaf(p.R, px, p.Ox) + offx;
            const float oy = fmaf(p.R, py, p.Oy) + offy;
            const float oz = fmaf(p.R, pz, p.Oz) + offz;

            // far end of the segment inside S: with f = o - O = R p + off and off . p = 0,
            // b = f . d and |f|^2 - R^2 = |off|^2
            const float b = fmaf(p.R, pd, fmaf(offx, dx, fmaf(offy, dy, offz * dz)));
            const float c = fmaf(offx, offx, fmaf(offy, offy, offz * offz));
            const float disc = fmaf(b, b, -c);
            const float t_end = disc > 0.0f ? fmaxf(0.0f, sqrtf(disc) - b) : 0.0f;

            const float4 r = march<BP, kPreUnroll>(p, ox, oy, oz, dx, dy, dz, t_end);
            acc0 += r.x;
            acc1 += r.y;
            acc2 += r.z;
            acc3 += r.w;
        }
        const float inv = 1.0f / (float)p.spp;
        if (p.C == 4) {
            reinterpret_cast<float4 *>(p.out)[t] = make_float4(acc0 * inv, acc1 * inv, acc2 * inv, acc3 * inv);
        } else {
            float *o = p.out + 3 * t;
            o[0] = acc0 * inv;
            o[1] = acc1 * inv;
            o[2] = acc2 * inv;
        }
    }
}

// Direct render of the same volume, one thread per pixel, in tiles of 16 x 16
// pixels and warps of 8 x 4 (the rays of a warp run side by side): the pixel's
// camera ray and its front hit h_o on S (the FP32 steps of the light-field
// render), the length of the ray inside S from h_o (chord_length), then the
// integral of the precompute along that ray (one sample, no jitter). Misses
// store 0. What bounds it, and the precompute: the FP32 pipe (70 and 73% of its
// cycles, with packed pairs at two cycles each), XU (54 and 59%) and issue (73%)
// together. 8 views of 512^2, 62% hit: 133 us; the chord in FP64, one launch a view
// and rows of 256 pixels took 241.
constexpr uint32_t kVolTileLog = 4;

template <int MAXV>
struct VolumeParams : PrecomputeParams {
    SphereK sphere;
    uint32_t n_views;
    uint32_t tile_prefix[MAXV + 1];
    ViewK views[MAXV];
};

template <int BP, int MAXV>
__global__ void __launch_bounds__(256, BP <= 4 ? kVolBlocks : 2)
    volume_direct_kernel(const __grid_constant__ VolumeParams<MAXV> p)
{
    uint32_t lo = 0, hi = p.n_views;                     // largest view with tile_prefix <= blockIdx.x
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (p.tile_prefix[mid] <= blockIdx.x) lo = mid; else hi = mid;
    }
    const ViewK &v = p.views[lo];
    const uint32_t lt = blockIdx.x - p.tile_prefix[lo];
    const uint32_t ty = (uint32_t)(((uint64_t)lt * v.div_m) >> v.div_s), tx = lt - ty * v.tiles_x;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t x = (tx << kVolTileLog) + ((warp & 1u) << 3) + (lane & 7u);
    const uint32_t y = (ty << kVolTileLog) + ((warp >> 1) << 2) + (lane >> 3);
    if (x >= v.width || y >= v.height) return;
    float4 r = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (!certain_miss(v, x, y)) {
        const float3 d = camera_dir(v, x, y);
        float3 ho, hd;
        if (intersect_sphere(p.sphere, v.eye, d, ho, hd))
            r = march<BP, kVolUnroll>(p, ho.x, ho.y, ho.z, d.x, d.y, d.z, chord_length(p.sphere, ho, d));
    }
    const uint64_t pix = v.out_offset + (uint64_t)y * v.width + x;
    if (p.C == 4) {
        reinterpret_cast<float4 *>(p.out)[pix] = r;
    } else {
        float *o = p.out + 3 * pix;
        o[0] = r.x;
        o[1] = r.y;
        o[2] = r.z;
    }
}

// One kernel per number of blob pairs: a scene of 3 blobs pays for 4, not 8, one
// of 9 for 10, not 16.
template <int MAXV>
static cudaError_t launch_volume(const VolumeParams<MAXV> &p, unsigned grid, cudaStream_t st)
{
    static const void *const f[] = {
        (const void *)volume_direct_kernel<1, MAXV>, (const void *)volume_direct_kernel<2, MAXV>,
        (const void *)volume_direct_kernel<3, MAXV>, (const void *)volume_direct_kernel<4, MAXV>,
        (const void *)volume_direct_kernel<5, MAXV>, (const void *)volume_direct_kernel<6, MAXV>,
        (const void *)volume_direct_kernel<7, MAXV>, (const void *)volume_direct_kernel<8, MAXV>};
    static_assert(kMaxBlobs == 16, "pairs");
    void *args[] = {const_cast<VolumeParams<MAXV> *>(&p)};
    return launch_kernel(f[p.nb ? (p.nb - 1) / 2 : 0], dim3(grid), 256, args, st);
}

static bool output_overlap(const ViewK &a, const ViewK &b)
{
    const uint64_t ea = a.out_offset + (uint64_t)a.width * a.height, eb = b.out_offset + (uint64_t)b.width * b.height;
    return a.out_offset < eb && b.out_offset < ea;
}

template <int MAXV>
static cudaError_t launch_views(const PrecomputeParams &base, const SphereK &S, const lf_view *views, uint32_t n,
                                double R, const double O[3], cudaStream_t st)
{
    static thread_local VolumeParams<MAXV> p;
    static_cast<PrecomputeParams &>(p) = base;
    p.sphere = S;
    lf_launch tile = {1u << kVolTileLog, 1u << kVolTileLog, 8, 0, 0, 0};
    for (uint32_t v0 = 0; v0 < n;) {
        // as many views as the parameters hold, a grid of fewer than 2^31 tiles, and no
        // view that overlaps an earlier one of the launch in the output: the last one
        // stays there, as if each view had its own launch
        uint64_t tiles = 0;
        uint32_t nv = 0;
        for (; nv < (uint32_t)MAXV && v0 + nv < n; ++nv) {
            p.views[nv] = view_params(views[v0 + nv], tile, R, O);
            const uint64_t t = (uint64_t)p.views[nv].tiles_x * p.views[nv].tiles_y;
            if (nv && tiles + t >= (1ull << 31)) break;
            bool overlaps = false;
            for (uint32_t k = 0; k < nv; ++k) overlaps |= output_overlap(p.views[k], p.views[nv]);
            if (overlaps) break;
            p.tile_prefix[nv] = (uint32_t)tiles;
            tiles += t;
        }
        p.n_views = nv;
        const cudaError_t e = launch_volume<MAXV>(p, (unsigned)tiles, st);
        if (e != cudaSuccess) return e;
        v0 += nv;
    }
    return cudaSuccess;
}

cudaError_t launch_volume_direct(const PrecomputeParams &p, const lf_view *views, uint32_t n, const SphereK &S, double R,
                                 const double O[3], cudaStream_t st)
{
    return n <= (uint32_t)kSmallViews ? launch_views<kSmallViews>(p, S, views, n, R, O, st)
                                      : launch_views<kVolumeViews>(p, S, views, n, R, O, st);
}

cudaError_t launch_precompute(const PrecomputeParams &p, cudaStream_t st)
{
    static const void *const f[] = {(const void *)precompute_kernel<1>, (const void *)precompute_kernel<2>,
                                    (const void *)precompute_kernel<3>, (const void *)precompute_kernel<4>,
                                    (const void *)precompute_kernel<5>, (const void *)precompute_kernel<6>,
                                    (const void *)precompute_kernel<7>, (const void *)precompute_kernel<8>};
    const uint64_t total = (uint64_t)p.rows * p.N;
    const uint64_t blocks = (total + 255) / 256;
    const unsigned grid = (unsigned)(blocks < (1ull << 20) ? blocks : (1ull << 20));
    void *args[] = {const_cast<PrecomputeParams *>(&p)};
    return launch_kernel(f[p.nb ? (p.nb - 1) / 2 : 0], dim3(grid), 256, args, st);
}

}  // namespace lfk
