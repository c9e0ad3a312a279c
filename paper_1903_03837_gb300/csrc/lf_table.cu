// lf_table.cu -- table-side kernels: the SF point caches, the per-row
// FP16/E4M3 quantiser, 3->4 channel padding of codes, and the synthetic lobe
// radiance field.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "lf_kernels.h"

namespace lfk {

// round(2^128 * (Phi - 1)) split into two 64-bit words: frac(i/Phi) =
// frac(i*(Phi-1)) is (i * G mod 2^128) / 2^128 up to i * 2^-129.
constexpr uint64_t kGoldHi = 0x9e3779b97f4a7c15ull;
constexpr uint64_t kGoldLo = 0xf39cc0605cedc834ull;
constexpr double kTwoPi = 6.283185307179586476925286766559;

// SF point p_i of a set of n points (Section 2, SF point set equation):
// phi_i = 2*pi*frac(i/Phi) (phase truncated to 53 bits), z_i = 1 - (2i+1)/n,
// p_i = (cos(phi_i) sin(theta_i), sin(phi_i) sin(theta_i), z_i) with
// sin(theta_i) = sqrt((1 - z_i)(1 + z_i)); FP64, stored as hi/lo floats and,
// when xy is given, as (x_hi, y_hi, x_lo, y_lo) between kPointPad far points on
// either side.
__global__ void build_points_kernel(uint32_t n, float4 *hi, float4 *lo, float4 *xy)
{
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (xy && i < 2u * kPointPad) xy[i < (uint32_t)kPointPad ? i : n + i] = make_float4(4.0f, 4.0f, 0.0f, 0.0f);
    if (i >= n) return;
    uint64_t ii = i;
    uint64_t top = ii * kGoldHi + __umul64hi(ii, kGoldLo);
    double t = (double)(top >> 11) * 0x1p-53;
    double phi = __dmul_rn(kTwoPi, t);
    double z = __dsub_rn(1.0, __ddiv_rn((double)(2ull * ii + 1ull), (double)n));
    double s = __dsqrt_rn(__dmul_rn(__dsub_rn(1.0, z), __dadd_rn(1.0, z)));
    double sp, cp;
    sincos(phi, &sp, &cp);
    double p[3] = {__dmul_rn(cp, s), __dmul_rn(sp, s), z};
    float h[3], l[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        h[k] = __double2float_rn(p[k]);
        l[k] = __double2float_rn(__dsub_rn(p[k], (double)h[k]));
    }
    hi[i] = make_float4(h[0], h[1], h[2], 0.0f);
    lo[i] = make_float4(l[0], l[1], l[2], 0.0f);
    if (xy) xy[kPointPad + i] = make_float4(h[0], h[1], l[0], l[1]);
}

cudaError_t launch_build_points(uint32_t n, float4 *hi, float4 *lo, float4 *xy, cudaStream_t st)
{
    build_points_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, hi, lo, xy);   // at least 2 kPointPad threads
    return cudaGetLastError();
}

// [M][N][3] codes -> [M][N][4] codes with channel 3 = 0.
template <typename T>
__global__ void pad_codes_kernel(const T *src, uint64_t texels, T *dst)
{
    uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= texels) return;
    dst[4 * t] = src[3 * t];
    dst[4 * t + 1] = src[3 * t + 1];
    dst[4 * t + 2] = src[3 * t + 2];
    dst[4 * t + 3] = T(0);
}

cudaError_t launch_pad_codes(const void *src, uint32_t M, uint32_t N, int bytes, void *dst, cudaStream_t st)
{
    uint64_t texels = (uint64_t)M * N;
    unsigned grid = (unsigned)((texels + 255) / 256);
    if (bytes == 2)
        pad_codes_kernel<<<grid, 256, 0, st>>>((const uint16_t *)src, texels, (uint16_t *)dst);
    else
        pad_codes_kernel<<<grid, 256, 0, st>>>((const uint8_t *)src, texels, (uint8_t *)dst);
    return cudaGetLastError();
}

// Per-row quantisation: amax over the row's N*C values; scale = amax (F16) or
// amax/448 (E4M3), 1 if amax = 0; codes of RNE(x / scale) (E4M3 saturating to
// +-448), 4 channels per texel.
__device__ __forceinline__ uint16_t e4m3x2(float a_hi, float b_lo)
{
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(a_hi), "f"(b_lo));
    return r;
}

// Scale of a row, and division by it. x / s is rounded to FP32 before the code is,
// so the quotient has to be the correctly rounded one: from the rounded reciprocal
// r of s, q0 = x r, and two steps q += (x - q s) r with the exact remainder (the
// first makes q faithful, the second correctly rounded: Markstein, "Computation
// of elementary functions on the IBM RISC System/6000 processor", 1990). The
// remainders are exact for s in [2^-60, 2^60] and quotients of 2^-26 and more;
// smaller ones have code 0 anyway. The sign is x's (a zero keeps it). Six
// instructions an element, where an IEEE division a value kept the issue slots 70%
// busy; other scales (denormal, infinite) take that.
struct RowScale {
    float s, r;
    bool direct;
};
template <int DTYPE>
__device__ __forceinline__ RowScale row_scale(float amax)
{
    RowScale c;
    c.s = amax == 0.0f ? 1.0f : (DTYPE == LF_DTYPE_E4M3 ? __fdiv_rn(amax, 448.0f) : amax);
    c.direct = !(c.s >= 0x1p-60f && c.s <= 0x1p60f);
    c.r = __frcp_rn(c.s);
    return c;
}
template <bool DIRECT>
__device__ __forceinline__ float over_scale(float x, const RowScale &c)
{
    if constexpr (DIRECT) return __fdiv_rn(x, c.s);
    float q = __fmul_rn(x, c.r);
    q = __fmaf_rn(__fmaf_rn(-q, c.s, x), c.r, q);
    q = __fmaf_rn(__fmaf_rn(-q, c.s, x), c.r, q);
    return copysignf(q, x);
}

// Code of a texel, as the 32 or 64 bits stored.
template <int DTYPE>
struct Code {
    using T = uint2;
    static __device__ __forceinline__ uint2 of(float x, float y, float z, float w)
    {
        __half2 a = __floats2half2_rn(x, y), b = __floats2half2_rn(z, w);
        return make_uint2(*reinterpret_cast<uint32_t *>(&a), *reinterpret_cast<uint32_t *>(&b));
    }
};
template <>
struct Code<LF_DTYPE_E4M3> {
    using T = uint32_t;
    static __device__ __forceinline__ uint32_t of(float x, float y, float z, float w)
    {
        return (uint32_t)e4m3x2(y, x) | ((uint32_t)e4m3x2(w, z) << 16);
    }
};

__device__ __forceinline__ float amax4(float m, float4 v)
{
    return fmaxf(fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
}

// Largest `v` over the row's threads: a warp, or a CTA of 8 warps.
template <int TPR>
__device__ __forceinline__ float row_max(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if constexpr (TPR > 32) {
        __shared__ float red[TPR / 32];
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
        __syncthreads();
        v = red[threadIdx.x & (TPR / 32 - 1)];
#pragma unroll
        for (int o = TPR / 64; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    }
    return v;
}

// The codes of a row held by TPR threads (quantize_held_kernel).
template <int DTYPE, int C, int TPR, int V, bool DIRECT>
__device__ __forceinline__ void store_held(const float4 (&x)[V][C == 4 ? 1 : 3], const RowScale &c, uint32_t i, uint32_t t,
                                           uint32_t units, typename Code<DTYPE>::T *codes)
{
    constexpr int W = C == 4 ? 1 : 3;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const uint32_t u = t + v * TPR;
        if (u >= units) continue;
        float q[4 * W];
#pragma unroll
        for (int k = 0; k < W; ++k) {
            q[4 * k] = over_scale<DIRECT>(x[v][k].x, c);
            q[4 * k + 1] = over_scale<DIRECT>(x[v][k].y, c);
            q[4 * k + 2] = over_scale<DIRECT>(x[v][k].z, c);
            q[4 * k + 3] = over_scale<DIRECT>(x[v][k].w, c);
        }
        if constexpr (C == 4) {
            codes[(size_t)i * units + u] = Code<DTYPE>::of(q[0], q[1], q[2], q[3]);
        } else {
            // four texels: 16 or 32 bytes
            typename Code<DTYPE>::T o[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) o[k] = Code<DTYPE>::of(q[3 * k], q[3 * k + 1], q[3 * k + 2], 0.0f);
            uint4 *d = reinterpret_cast<uint4 *>(codes) + ((size_t)i * units + u) * (sizeof o / 16);
#pragma unroll
            for (int k = 0; k < (int)(sizeof o / 16); ++k) d[k] = reinterpret_cast<const uint4 *>(o)[k];
        }
    }
}

// Rows held in registers between the maximum and the codes, so the table is read
// once, 16 bytes a load. A unit is one RGBA texel, or four RGB texels (48 bytes);
// a row is V units for each of TPR threads (a warp for short rows, else the CTA).
// 65,536 rows of 1,024 RGBA texels to E4M3: 0.191 ms, bound by HBM (1.34 GB at 7.0
// TB/s); two passes of scalar loads with IEEE divisions took 0.314. Rows of 100
// texels: 5.7 times as fast as a CTA each; of 4,096: 1.6 times as the two passes.
// 4 to 6 CTAs per SM for 16 floats a thread are alike, 8 (spilling) 2% slower.
template <int DTYPE, int C, int TPR, int V>
__global__ void __launch_bounds__(256, V * (C == 4 ? 1 : 3) <= 4 ? 6 : V * (C == 4 ? 1 : 3) <= 8 ? 4 : 2)
    quantize_held_kernel(const float4 *src, uint32_t M, uint32_t units,
                                                            typename Code<DTYPE>::T *codes, float *scales)
{
    constexpr int W = C == 4 ? 1 : 3;                    // float4 per unit
    const uint32_t i = TPR == 32 ? blockIdx.x * 8 + (threadIdx.x >> 5) : blockIdx.x, t = threadIdx.x & (TPR - 1);
    if (TPR == 32 && i >= M) return;                     // whole warps
    const float4 *r = src + (size_t)i * units * W;
    float4 x[V][W];
    float amax = 0.0f;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const uint32_t u = t + v * TPR;
#pragma unroll
        for (int k = 0; k < W; ++k) x[v][k] = u < units ? __ldcs(r + (size_t)u * W + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int k = 0; k < W; ++k) amax = amax4(amax, x[v][k]);
    const RowScale c = row_scale<DTYPE>(row_max<TPR>(amax));
    if (t == 0) scales[i] = c.s;
    if (c.direct)                                        // the same in the whole row
        store_held<DTYPE, C, TPR, V, true>(x, c, i, t, units, codes);
    else
        store_held<DTYPE, C, TPR, V, false>(x, c, i, t, units, codes);
}

// Rows too long for the registers, unaligned buffers, and RGB rows that are not a
// whole number of four texels: two passes, one CTA per row.
template <int DTYPE>
__global__ void quantize_rows_kernel(const float *src, uint32_t N, uint32_t C, void *codes, float *scales)
{
    const uint32_t i = blockIdx.x;
    const size_t rowlen = (size_t)N * C;
    const float *r = src + (size_t)i * rowlen;
    float amax = 0.0f;
    // 16-byte loads from the row's first aligned float on
    const uint32_t head = min((uint32_t)rowlen, (uint32_t)((16 - ((uintptr_t)r & 15)) & 15) / 4);
    const size_t quads = (rowlen - head) / 4;
    const float4 *r4 = reinterpret_cast<const float4 *>(r + head);
    for (size_t k = threadIdx.x; k < quads; k += blockDim.x) amax = amax4(amax, r4[k]);
    if (threadIdx.x < head) amax = fmaxf(amax, fabsf(r[threadIdx.x]));
    const size_t tail = head + 4 * quads + threadIdx.x;
    if (tail < rowlen) amax = fmaxf(amax, fabsf(r[tail]));
    const RowScale c = row_scale<DTYPE>(row_max<256>(amax));
    if (threadIdx.x == 0) scales[i] = c.s;
    typename Code<DTYPE>::T *o = reinterpret_cast<typename Code<DTYPE>::T *>(codes) + (size_t)i * N;
    const bool vec = C == 4 && head == 0;
    for (uint32_t j = threadIdx.x; j < N; j += blockDim.x) {
        float4 x;
        if (vec) {
            x = r4[j];
        } else {
            const float *q = r + (size_t)j * C;
            x = make_float4(q[0], q[1], q[2], C == 4 ? q[3] : 0.0f);
        }
        if (c.direct)
            o[j] = Code<DTYPE>::of(over_scale<true>(x.x, c), over_scale<true>(x.y, c), over_scale<true>(x.z, c),
                                   over_scale<true>(x.w, c));
        else
            o[j] = Code<DTYPE>::of(over_scale<false>(x.x, c), over_scale<false>(x.y, c), over_scale<false>(x.z, c),
                                   over_scale<false>(x.w, c));
    }
}

template <int DTYPE, int C, int TPR, int V>
static void launch_held(const float *src, uint32_t M, uint32_t units, void *codes, float *scales, cudaStream_t st)
{
    const unsigned grid = TPR == 32 ? (M + 7) / 8 : M;
    quantize_held_kernel<DTYPE, C, TPR, V><<<grid, 256, 0, st>>>(reinterpret_cast<const float4 *>(src), M, units,
                                                                 reinterpret_cast<typename Code<DTYPE>::T *>(codes), scales);
}

// The registers hold rows of up to 4,096 texels (64 floats a thread); up to 256
// texels a warp holds a row, which needs no barrier.
template <int DTYPE>
static void launch_quantize_as(const float *src, uint32_t M, uint32_t N, uint32_t C, void *codes, float *scales,
                               cudaStream_t st)
{
    const bool aligned = ((uintptr_t)src & 15) == 0 && ((uintptr_t)codes & 15) == 0;
    const uint32_t u = C == 4 ? N : N / 4;
    if (aligned && C == 4 && N <= 4096) {
        if (u <= 64) launch_held<DTYPE, 4, 32, 2>(src, M, u, codes, scales, st);
        else if (u <= 128) launch_held<DTYPE, 4, 32, 4>(src, M, u, codes, scales, st);
        else if (u <= 256) launch_held<DTYPE, 4, 32, 8>(src, M, u, codes, scales, st);
        else if (u <= 512) launch_held<DTYPE, 4, 256, 2>(src, M, u, codes, scales, st);
        else if (u <= 1024) launch_held<DTYPE, 4, 256, 4>(src, M, u, codes, scales, st);
        else if (u <= 2048) launch_held<DTYPE, 4, 256, 8>(src, M, u, codes, scales, st);
        else launch_held<DTYPE, 4, 256, 16>(src, M, u, codes, scales, st);
    } else if (aligned && C == 3 && N % 4 == 0 && N <= 4096) {
        if (u <= 32) launch_held<DTYPE, 3, 32, 1>(src, M, u, codes, scales, st);
        else if (u <= 64) launch_held<DTYPE, 3, 32, 2>(src, M, u, codes, scales, st);
        else if (u <= 256) launch_held<DTYPE, 3, 256, 1>(src, M, u, codes, scales, st);
        else if (u <= 512) launch_held<DTYPE, 3, 256, 2>(src, M, u, codes, scales, st);
        else launch_held<DTYPE, 3, 256, 4>(src, M, u, codes, scales, st);
    } else {
        quantize_rows_kernel<DTYPE><<<M, 256, 0, st>>>(src, N, C, codes, scales);
    }
}

cudaError_t launch_quantize(const float *src, uint32_t M, uint32_t N, uint32_t C, int dtype, void *codes,
                            float *scales, cudaStream_t st)
{
    if (dtype == LF_DTYPE_E4M3)
        launch_quantize_as<LF_DTYPE_E4M3>(src, M, N, C, codes, scales, st);
    else
        launch_quantize_as<LF_DTYPE_F16>(src, M, N, C, codes, scales, st);
    return cudaGetLastError();
}

__device__ __forceinline__ double dot3(const double a[3], const double b[3])
{
    return __dadd_rn(__dadd_rn(__dmul_rn(a[0], b[0]), __dmul_rn(a[1], b[1])), __dmul_rn(a[2], b[2]));
}

// Lobe field, one thread per texel (i, j); a CTA covers 256 columns of one row
// and shares that row's position factors. FP64, rounded once to FP32.
__global__ void fill_lobe_kernel(const __grid_constant__ LobeParams P, const float4 *po_hi,
                                 const float4 *po_lo, const float4 *pd_hi, const float4 *pd_lo,
                                 uint32_t N, uint32_t blocks_per_row, float *out)
{
    __shared__ double s_ep[kMaxLobes];
    const uint32_t i = blockIdx.x / blocks_per_row;
    const uint32_t j = (blockIdx.x % blocks_per_row) * blockDim.x + threadIdx.x;
    float4 a = po_hi[i], b = po_lo[i];
    const double po[3] = {__dadd_rn((double)a.x, (double)b.x), __dadd_rn((double)a.y, (double)b.y),
                          __dadd_rn((double)a.z, (double)b.z)};
    if (threadIdx.x < P.L) {
        double cp = dot3(po, P.ap[threadIdx.x]);
        s_ep[threadIdx.x] = exp(__dmul_rn(P.kp[threadIdx.x], __dsub_rn(cp, 1.0)));
    }
    __syncthreads();
    if (j >= N) return;
    float4 c = pd_hi[j], e = pd_lo[j];
    double d[3] = {__dsub_rn(__dadd_rn((double)c.x, (double)e.x), po[0]),
                   __dsub_rn(__dadd_rn((double)c.y, (double)e.y), po[1]),
                   __dsub_rn(__dadd_rn((double)c.z, (double)e.z), po[2])};
    double l = __dsqrt_rn(dot3(d, d));
    if (l < 1e-12) {
        d[0] = -po[0]; d[1] = -po[1]; d[2] = -po[2];
    } else {
        d[0] = __ddiv_rn(d[0], l); d[1] = __ddiv_rn(d[1], l); d[2] = __ddiv_rn(d[2], l);
    }
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (uint32_t k = 0; k < P.L; ++k) {
        double cd = dot3(d, P.ad[k]);
        double g = __dmul_rn(s_ep[k], exp(__dmul_rn(P.kd[k], __dsub_rn(cd, 1.0))));
        for (uint32_t ch = 0; ch < P.C; ++ch) acc[ch] = __dadd_rn(acc[ch], __dmul_rn(P.col[k][ch], g));
    }
    float *o = out + ((size_t)i * N + j) * P.C;
    for (uint32_t ch = 0; ch < P.C; ++ch) {
        uint64_t ctr = ((uint64_t)i << 32) | ((uint64_t)j << 4) | ch;
        double u = (double)(splitmix64(P.seed, ctr) >> 11) * 0x1p-53;
        o[ch] = __double2float_rn(__dadd_rn(acc[ch], __dmul_rn(0.01, u)));
    }
}

cudaError_t launch_fill_lobe(const LobeParams &P, const float4 *po_hi, const float4 *po_lo,
                             const float4 *pd_hi, const float4 *pd_lo, uint32_t M, uint32_t N,
                             float *out, cudaStream_t st)
{
    uint32_t bpr = (N + 255) / 256;
    fill_lobe_kernel<<<(unsigned)((uint64_t)M * bpr), 256, 0, st>>>(P, po_hi, po_lo, pd_hi, pd_lo, N, bpr, out);
    return cudaGetLastError();
}

}  // namespace lfk
