// lf_render.cu -- forward render kernels of the light-field sampling path
// (LumiPath, arXiv 1903.03837, Section 2).
//
// One thread per camera ray. A CTA renders a tile of tile_w x tile_h pixels of
// one view; each warp covers a warp_w x (32/warp_w) sub-tile so that its rays
// hit neighbouring SF cells and share texels in L1. Tiles of all views of a
// call are numbered consecutively (view-major), one CTA per tile: the hardware's
// block scheduler hands them out. Views live in the kernel's parameter space (no
// device copy, graph friendly), and a CTA's view and tile depend on blockIdx
// alone, so their fields are read through uniform registers. A persistent grid
// that pulled tiles from a queue word read them through per-lane constant loads
// instead, one barrier and one shared word per tile: 18% slower on 64 uneven
// views (4.10 against 3.46 ms), so a launch is never persistent.
//
// What bounds it: instruction issue (79% of the issue slots on a 1080p frame of
// a 65,536 x 1,024 FP16 table, ALU pipe 48%, FMA 39%, DRAM 3%). An image lists
// the points within the kernel's radius (lf_ray.cuh) instead of ranking the
// nearest ones and certifying the order: that frame 0.050 ms instead of 0.119
// (1,420 thread instructions per hit ray instead of 2,680, and no exact pass), a
// 2 x 3840 x 2160 frame of a 262,144 x 4,096 E4M3 table 0.258 instead of 0.547,
// 64 uneven views of a 16,384 x 512 FP16 table 3.29 instead of 6.46. Per hit ray of
// that frame, counted before the corners' z differences were rounded once: blend
// 381, candidates' distances 250, lattice corners 267, unit hits 182, camera and
// hits 107, lists 76.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "lf_ray.cuh"

// Resident CTAs of kMaxBlock threads per SM the register budget of the unranked
// kernels is cut for: 5 (48 registers, 12 to 24 bytes spilled) against 4 took the 4K
// stereo frame from 277 to 252 us and the 64 views from 3.29 to 3.19 ms; 6 was 2%
// slower than 5. The variants that rank 5 indices spill 130 bytes at 4.
#ifndef LF_MIN_BLOCKS
#define LF_MIN_BLOCKS 5
#endif

namespace lfk {

// Byte size of a stored texel.
template <int DT>
constexpr uint32_t kTexelBytes = DT == kF32C4 ? 16 : DT == kF32C3 ? 12 : DT == kF16C4 ? 8 : 4;

// Texel at byte offset `off` of the table (its channels to FP32).
template <int DT, typename Off>
__device__ __forceinline__ float4 texel_at(const RenderParamsBase &p, Off off)
{
#ifdef LF_DEBUG_CHECKS
    off = (Off)LF_DINDEX((uint64_t)off / kTexelBytes<DT>, (uint64_t)p.rows_valid * p.N, p.status, kStatusDebugTexel) *
          kTexelBytes<DT>;
#endif
    const char *q = reinterpret_cast<const char *>(p.texels) + off;
    if constexpr (DT == kF32C3) {
        // 12-byte texels as the 8-byte-aligned pair and the remaining float
        const bool odd = ((uint32_t)off & 4u) != 0;
        const float2 pair = __ldg(reinterpret_cast<const float2 *>(q + (odd ? 4 : 0)));
        const float one = __ldg(reinterpret_cast<const float *>(q + (odd ? 0 : 8)));
        return odd ? make_float4(one, pair.x, pair.y, 0.0f) : make_float4(pair.x, pair.y, one, 0.0f);
    } else {
        return texel<DT>(q, 0);
    }
}

struct RayLists {
    uint2 e[2][kListSlots][kMaxBlock];
};

// Blend of one ray's listed origins and directions: sum of w_a w_b texel / (sum
// w_a)(sum w_b). The loop over origins runs to the longest list of the warp and
// the fifth direction (0.3% of rays have one) sits behind a branch of the warp;
// up to there a lane without a neighbour reads its first direction's column (a
// texel it loads anyway) with weight 0: a branch around the load costs more than
// the load. Every texel is finite (the FP32 table is the caller's promise; FP16
// and E4M3 codes are finite by construction), so such a tap adds exactly 0. The
// direction weights are a quarter of the tent: a set's weights sum to at most 1.32,
// so every sum stays below 0.44 of the largest texel and cannot overflow (an
// infinite sum times the weight 0 of an origin slot past the list would be NaN). A
// power of two changes no bit of the quotient and takes no instruction.
// Every lane of the warp calls it.
template <int DT, typename Off>
__device__ __forceinline__ float4 blend(const RenderParamsBase &p, const RayLists &L, int co, int cd)
{
    const unsigned most = __reduce_or_sync(0xffffffffu, (1u << co) | (0x100u << cd));
    const int co_w = 31 - __clz(most & 0xffu);           // longest lists of the warp
    const bool five = (most >> (8 + kListSlots)) != 0;
    if (co_w == 0) return make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    Off jo[kListSlots];
    float wd[kListSlots], sd = 0.0f;
#pragma unroll
    for (int b = 0; b < kListSlots; ++b) {
        wd[b] = 0.0f;
        if (b == kListSlots - 1 && !five) break;
        const uint2 e = L.e[1][b][threadIdx.x];
        const bool live = b < cd;
        jo[b] = b == 0 ? (live ? e.x * kTexelBytes<DT> : 0u) : (live ? (Off)(e.x * kTexelBytes<DT>) : jo[0]);
        wd[b] = live ? quarter_tent(__uint_as_float(e.y), p.pd.inv_sigma) : 0.0f;
        sd += wd[b];
    }
    float2 acc_xy = make_float2(0.f, 0.f), acc_zw = make_float2(0.f, 0.f);
    float so = 0.0f;
#pragma unroll 1
    for (int a = 0; a < co_w; ++a) {
        const uint2 e = L.e[0][a][threadIdx.x];
        const bool live = a < co;
        const uint32_t i = live ? e.x : 0u;
        const float w = live ? tent(__uint_as_float(e.y), p.po.inv_sigma) : 0.0f;
        so += w;
        float s = w;
        if constexpr (DT == kF16C4 || DT == kE4M3C4) s *= __ldg(p.scales + i);
        const Off row = (Off)i * ((Off)p.N * (Off)kTexelBytes<DT>);
        float2 in_xy, in_zw;
#pragma unroll
        for (int b = 0; b < kListSlots; ++b) {
            if (b == kListSlots - 1 && !five) break;
            const float4 t = texel_at<DT, Off>(p, row + jo[b]);
            const float2 w2 = make_float2(wd[b], wd[b]);
            in_xy = ffma2(w2, make_float2(t.x, t.y), b ? in_xy : make_float2(0.f, 0.f));
            in_zw = ffma2(w2, make_float2(t.z, t.w), b ? in_zw : make_float2(0.f, 0.f));
        }
        const float2 s2 = make_float2(s, s);
        acc_xy = ffma2(s2, in_xy, acc_xy);
        acc_zw = ffma2(s2, in_zw, acc_zw);
    }
    const float r = co ? rcp_approx(so * sd) : 0.0f;
    return make_float4(acc_xy.x * r, acc_xy.y * r, acc_zw.x * r, acc_zw.y * r);
}

template <int DT, int IDX, typename Off>
__device__ __forceinline__ void render_ray(const RenderParamsBase &p, const ViewK &v, uint32_t vi, bool active,
                                           uint32_t px, uint32_t py, RayLists &L)
{
    constexpr int KI = IDX ? IDX : 1;
    int32_t io[KI], jd[KI];
    int co = 0, cd = 0;
    uint32_t pend = 0;
    bool hit = active && !certain_miss(v, px, py) &&
               ray_lists<IDX, kMaxBlock>(p, v, camera_dir(v, px, py), &L.e[0][0][threadIdx.x], co, cd, io, jd, pend);
    if (!hit || (pend & kPendImage)) co = cd = 0;
    const float4 acc = blend<DT, Off>(p, L, co, cd);
    if (!active) return;
    if (pend) defer_push(p, vi, px, py, pend);
    if (pend & kPendImage) return;
    const uint64_t pix = pixel_index(v, px, py);
    store_image(p, pix, acc);
    if constexpr (IDX != 0) {
        if (!p.idx || pend) return;                      // pend: the fixup kernel writes the indices
        if (!hit) {
#pragma unroll
            for (int m = 0; m < KI; ++m) io[m] = jd[m] = -1;
        }
        store_idx<KI>(p, pix, io, jd);
    } else if (p.idx) {                                  // nearest sampling: the listed point of each set
        const int32_t i = hit ? (int32_t)L.e[0][0][threadIdx.x].x : -1, j = hit ? (int32_t)L.e[1][0][threadIdx.x].x : -1;
        reinterpret_cast<int2 *>(p.idx)[pix] = make_int2(i, j);
    }
}

// A pixel of a tile outside the view's screen bound of S. (One warp storing the
// whole tile while the others leave takes fewer instructions and more time: 9% on
// the 4K stereo frame, 59% of whose tiles miss.)
template <int IDX>
__device__ __forceinline__ void store_miss(const RenderParamsBase &p, const ViewK &v, uint32_t px, uint32_t py)
{
    const uint64_t pix = pixel_index(v, px, py);
    store_image(p, pix, make_float4(0.0f, 0.0f, 0.0f, 0.0f));
    if (p.idx) {
        constexpr int KI = IDX ? IDX : 1;
        int32_t none[KI];
#pragma unroll
        for (int m = 0; m < KI; ++m) none[m] = -1;
        store_idx<KI>(p, pix, none, none);
    }
}

template <int DT, int MAXV, int IDX, typename Off>
__global__ void __launch_bounds__(kMaxBlock, IDX == 9 ? 2 : IDX == 5 ? 4 : LF_MIN_BLOCKS)
    render_kernel(const __grid_constant__ RenderParams<MAXV> p)
{
    __shared__ RayLists L;
    uint32_t v, tx, ty, px, py;        // v, tx, ty: the same in the whole CTA (uniform registers)
    if (!cta_tile(p, v, tx, ty)) return;
    const ViewK &vw = p.views[v];
    pixel_of(p, tx, ty, px, py);
    const bool active = px < vw.width && py < vw.height;
    if (tile_misses(p, vw, tx, ty)) {
        if (active) store_miss<IDX>(p, vw, px, py);
    } else {
        render_ray<DT, IDX, Off>(p, vw, v, active, px, py, L);
    }
}

// The kernel of a launch. Indices (5 or 9 neighbours) take the ranked variants;
// an upper-hemisphere table with nine neighbours too, whose masked rays need the
// 9 nearest. Nearest sampling and images alone take the unranked one, with
// 32-bit texel offsets while the table is at most 4 GiB.
template <int DT, int MAXV>
static const void *render_fn(const RenderParamsBase &p)
{
    if (p.nine && (p.idx || p.rows_stored)) return (const void *)render_kernel<DT, MAXV, 9, uint64_t>;
    if (p.idx && !p.nearest_only) return (const void *)render_kernel<DT, MAXV, 5, uint64_t>;
    return p.table_bytes <= (1ull << 32) ? (const void *)render_kernel<DT, MAXV, 0, uint32_t>
                                         : (const void *)render_kernel<DT, MAXV, 0, uint64_t>;
}

template <int MAXV>
static const void *render_fn(int kind, const RenderParamsBase &p)
{
    switch (kind) {
    case kF32C4: return render_fn<kF32C4, MAXV>(p);
    case kF32C3: return render_fn<kF32C3, MAXV>(p);
    case kF16C4: return render_fn<kF16C4, MAXV>(p);
    default: return render_fn<kE4M3C4, MAXV>(p);
    }
}

// Whether a launch may queue rays: 5-neighbour indices and nearest sampling
// leave near-ties to the exact pass, upper-hemisphere tables the rays at the
// rim of their rows; an image of 5 or 9 neighbours never does.
static bool may_defer(const RenderParamsBase &p)
{
    if (p.nine) return false;
    return p.nearest_only || p.idx != nullptr || p.rows_stored != 0;
}

template <int MAXV>
static cudaError_t launch(int kind, const RenderParams<MAXV> &p, dim3 grid, unsigned block, cudaStream_t st)
{
    void *args[] = {const_cast<RenderParams<MAXV> *>(&p)};
    cudaError_t e = launch_kernel(render_fn<MAXV>(kind, p), grid, block, args, st);
    if (e == cudaSuccess && may_defer(p)) e = launch_fixup(kind, false, p, st);
    return e;
}

cudaError_t launch_render(int kind, const RenderParams<kSmallViews> &p, dim3 grid, unsigned block, cudaStream_t st)
{
    return launch(kind, p, grid, block, st);
}
cudaError_t launch_render(int kind, const RenderParams<kLargeViews> &p, dim3 grid, unsigned block, cudaStream_t st)
{
    return launch(kind, p, grid, block, st);
}

}  // namespace lfk
