// lf_df.cuh -- double-float arithmetic, the z differences between a hit and the
// points of its lattice corners, and the length of a ray inside S. IEEE FP32 operations only, so a host compiler gives
// the same bits.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "lf_internal.h"

namespace lfk {

// ---------------------------------------------------------------------------
// Double-float arithmetic (value = hi + lo, about 48 significant bits).
// ---------------------------------------------------------------------------
struct df { float h, l; };
__device__ __forceinline__ df two_sum(float a, float b)
{
    float s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
__device__ __forceinline__ df fast_two_sum(float a, float b)
{
    float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ df df_add(df x, df y)
{
    df s = two_sum(x.h, y.h);
    return fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(x.l, y.l)));
}
__device__ __forceinline__ df df_mul(df x, df y)
{
    float p = __fmul_rn(x.h, y.h);
    float e = __fmaf_rn(x.h, y.h, -p);
    e = __fmaf_rn(x.h, y.l, __fmaf_rn(x.l, y.h, e));
    return fast_two_sum(p, e);
}

// ---------------------------------------------------------------------------
// q_z - z_i of a unit hit and the SF points around it (z_i = z_0 - i 2/n, z_0 = 1 - 1/n).
//
// For point b as c + r: c a multiple of the set's grid (about 2^-11 of the z step
// 2/n), r the rest, with every cancelling step exact. The corner k = i - b indices
// on then is (c + k zstep_c) + (r + k zstep_r): zstep_c is the step rounded to
// 11 bits, so the first sum is exact and the difference is rounded once, as the
// difference from a cached z is. Adding rounded multiples of the step instead is
// faster by 2% of a render (4K stereo frame 253 against 258 us), with tent weights
// off by up to 2.5e-7 for 1,000 points (rms 5.3e-8) where the cached z gives 1.7e-7
// (3.8e-8) and this 1.6e-7 (3.8e-8). Packed pairs of corners gain nothing.
// ---------------------------------------------------------------------------
struct ZOffset {
    float c, r;
};
__device__ __forceinline__ ZOffset z_offset(const PointSetK &P, int32_t b, float qzh, float qzl)
{
    const float bf = __int2float_rn(b);                  // exact: b <= 2^24
    const float t = __fmul_rn(bf, P.zstep_h);
    const float e = __fadd_rn(__fmaf_rn(bf, P.zstep_h, -t), __fmaf_rn(bf, P.zstep_l, -P.z0_l));
    const df s = two_sum(t, -P.z0_h);
    const float h = __fadd_rn(qzh, s.h);
    ZOffset o;
    o.c = __fsub_rn(__fadd_rn(h, P.zgrid), P.zgrid);
    o.r = __fadd_rn(__fsub_rn(h, o.c), __fadd_rn(__fadd_rn(qzl, s.l), e));
    return o;
}
__device__ __forceinline__ float z_at(const PointSetK &P, const ZOffset &o, float k)
{
    return __fadd_rn(__fmaf_rn(k, P.zstep_c, o.c), __fmaf_rn(k, P.zstep_r, o.r));
}

// ---------------------------------------------------------------------------
// Far end of the segment inside S from the front hit h along unit d: with f = h -
// O, b = f . d and c = |f|^2 - R^2, -b + sqrt(b^2 - c). In FP32, c cancels for a
// hit on S and b for a grazing ray; here every step up to the result is carried in
// double-float (c by the error-free expansion of unit_hit_df, the root by one Newton
// step), so the length is rounded once, as in FP64: relative error at most 6.0e-8
// (with b, c and the root each rounded to FP32 before the difference it was 1.3e-7).
// The same in FP64 costs some forty operations and a square root at a seventieth of
// FP32's rate.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float chord_length(const SphereK &S, float3 h, float3 d)
{
    const float hv[3] = {h.x, h.y, h.z}, dv[3] = {d.x, d.y, d.z};
    df b{0.0f, 0.0f}, sq{0.0f, 0.0f};
    float small = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const df s = two_sum(hv[k], -S.o_hi[k]);
        const df f = fast_two_sum(s.h, __fsub_rn(s.l, S.o_lo[k]));
        b = df_add(b, df_mul(f, df{dv[k], 0.0f}));
        const float p = __fmul_rn(f.h, f.h);
        small = __fadd_rn(small, __fmaf_rn(2.0f * f.h, f.l, __fmaf_rn(f.h, f.h, -p)));
        const df t = two_sum(sq.h, p);
        sq.h = t.h;
        sq.l = __fadd_rn(sq.l, t.l);
    }
    const df r = two_sum(sq.h, -S.r2_h);
    const df c = two_sum(r.h, __fadd_rn(__fadd_rn(r.l, sq.l), __fsub_rn(small, S.r2_l)));
    const float p = __fmul_rn(b.h, b.h);
    const df q = two_sum(p, -c.h);
    const df disc = fast_two_sum(
        q.h, __fadd_rn(q.l, __fsub_rn(__fmaf_rn(2.0f * b.h, b.l, __fmaf_rn(b.h, b.h, -p)), c.l)));
    if (!(disc.h > 0.0f)) return 0.0f;
    const float w = __fsqrt_rn(disc.h);
    const float wl = __fmul_rn(__fadd_rn(__fmaf_rn(-w, w, disc.h), disc.l), __fmul_rn(0.5f, __frcp_rn(w)));
    const df t = two_sum(w, -b.h);
    return fmaxf(0.0f, __fadd_rn(t.h, __fadd_rn(t.l, __fsub_rn(wl, b.l))));
}

}  // namespace lfk
