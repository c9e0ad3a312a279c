// lf_internal.h -- structures shared by the host side of the C ABI and the
// kernels of the light-field sampling library.
#pragma once

#include <stdint.h>

#include <cmath>

#include "lumipath.h"

namespace lfk {

// Bits of a table's device status word (read back by lf_sync_status).
constexpr uint32_t kStatusIndex = 1u;        // a search returned an index out of range (recorded, replaced by 0)
constexpr uint32_t kStatusIdxInput = 2u;     // given indices disagree with the ray (backward from indices)
constexpr uint32_t kStatusDebugPoint = 4u;   // debug build: a point index about to be read is out of range
constexpr uint32_t kStatusDebugTexel = 8u;   // debug build: a texel index about to be read is out of range
constexpr uint32_t kStatusDebugGrad = 16u;   // debug build: a gradient index about to be written is out of range

// Debug builds (-DLF_DEBUG_CHECKS), in place of a sanitizer: every index the
// kernels are about to dereference is checked against its bound; a failure
// sets a status bit and the access goes to index 0 instead (recorded, never a
// trap or a fault). Release builds: the index as it is (in range by construction).
#ifdef LF_DEBUG_CHECKS
#define LF_DINDEX(idx, bound, status, bit) \
    (((uint64_t)(idx) < (uint64_t)(bound)) ? (idx) : (atomicOr((status), (bit)), decltype(+(idx))(0)))
#else
#define LF_DINDEX(idx, bound, status, bit) (idx)
#endif

// Storage forms the kernels read (texel type x channel count).
enum TexelKind { kF32C4 = 0, kF32C3 = 1, kF16C4 = 2, kE4M3C4 = 3 };

// A view as the kernels read it (kernel-parameter space).
struct ViewK {
    float eye[3], right[3], up[3], fwd[3];
    float tan_x, tan_y;
    uint32_t width, height;
    uint64_t out_offset;
    uint32_t tiles_x, tiles_y;
    // Conservative miss test: e - O, |e - O|^2 - R^2, |e - O|^2, 2/W, 2/H
    // (host FP64, rounded), and whether the eye is clearly outside S.
    float f0[3], c0, ff0, inv2w, inv2h;
    uint32_t outside;
    float q[6];              // certain_miss: q0 + q1 x + q2 y + q3 x^2 + q4 x y + q5 y^2 < 0 at pixel (x, y)
    // Pixels outside columns [sx0, sx1) or rows [sy0, sy1) certainly miss S
    // (the screen bound of certain_miss, widened by three pixels).
    uint32_t sx0, sx1, sy0, sy1;
    // lt / tiles_x for any lt < 2^31 is (lt * div_m) >> div_s (64-bit product)
    uint32_t div_m, div_s;
};

// Sphere S: FP32 centre and radius for the ray/sphere step, the centre as a
// hi/lo float pair and in FP64 for the unit hit vectors.
struct SphereK {
    float o32[3];
    float r32;
    float o_hi[3], o_lo[3];
    double o64[3];
    float ir_h, ir_l;        // 1/R as a hi/lo pair
    float r2_h, r2_l;        // R^2 as a hi/lo pair
    float inv_r2;            // 1/R^2
    uint32_t centred;        // O == (0, 0, 0)
};

// Entries of the xy cache before point 0 and after point n - 1: points far from
// S, which a lattice corner outside the index range reads.
constexpr int32_t kPointPad = 64;

// One SF point set: p_i as hi/lo float4 pairs (w unused) and, for the searches
// that need x and y only (z is linear in i), as one float4 (x_hi, y_hi, x_lo,
// y_lo) at entry kPointPad + i; n, n as float, the kernel radius sigma = sqrt(4*pi/n) as its
// reciprocal and square (less 2^-20 of it), and the z step 2/n and z_0 = 1 - 1/n as hi/lo pairs.
struct PointSetK {
    const float4 *hi;
    const float4 *lo;
    const float4 *xy;
    uint32_t n;
    float nf, nhalf;         // n and n/2
    float zpole;             // |z| beyond which points_within scans (8 indices off a pole, or always)
    float inv_sigma;
    float sigma2;
    float zone0;             // log_{Phi^2}(sqrt5*pi*n), the set's part of the zone number
    float zstep_h, zstep_l, z0_h, z0_l;
    float zstep_c, zstep_r;  // the z step as 11 bits and the rest
    float zgrid;             // 1.5 2^23 units of the last of those bits: adding and taking it off rounds to them
};

inline void fill_z_steps(PointSetK &P)
{
    const double step = 2.0 / (double)P.n;
    int e;
    std::frexp(step, &e);
    const double unit = std::ldexp(1.0, e - 11);
    P.zstep_h = (float)step;
    P.zstep_l = (float)(step - (double)P.zstep_h);
    P.z0_h = (float)(1.0 - 0.5 * step);
    P.z0_l = (float)(1.0 - 0.5 * step - (double)P.z0_h);
    P.zstep_c = (float)(std::rint(step / unit) * unit);
    P.zstep_r = (float)(step - (double)P.zstep_c);
    P.zgrid = (float)std::ldexp(1.5 * unit, 23);
}

// Argument checks and view set-up shared by the entry points (lf_abi.cu): a
// failed check sets the calling thread's lf_last_error() message.
lf_status check_desc(const lf_table_desc *d);
lf_status check_launch(const lf_launch *c);
lf_status check_views(const lf_view *views, uint32_t n);
ViewK camera_of(const lf_view &w);                  // the camera only (no tiling, no miss constants)
ViewK view_params(const lf_view &w, const lf_launch &L, double R, const double O[3]);
// The set of n points with caches hi [n], lo [n], xy [n + 2 kPointPad].
PointSetK point_set_of(const float4 *hi, const float4 *lo, const float4 *xy, uint32_t n);

}  // namespace lfk

struct lf_table {
    lf_table_desc desc;
    int device;
    int texel_kind;                  // lfk::TexelKind
    uint32_t C;                      // logical channels (3 or 4)
    uint32_t rows;                   // origin rows stored (M, or M/2 for the upper hemisphere)
    const void *texels;              // [M][N][Cs]
    const float *scales;             // [M] or NULL (F32)
    void *owned_texels;              // non-NULL if the library owns the copy
    float *owned_scales;
    float4 *points;                  // origins hi, lo, xy, then directions hi, lo, xy
    uint32_t *scratch;               // device words and the queue of deferred rays (layout: lf_kernels.h)
    lfk::SphereK sphere;
    lfk::PointSetK po, pd;
    lf_launch launch;
};
