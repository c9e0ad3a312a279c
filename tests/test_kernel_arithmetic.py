"""The kernels' extended-precision arithmetic (csrc/lf_df.cuh), compiled here for the
host: it uses IEEE FP32 operations only, so the host gives the device's bits. Each
result against 64 bits or better, with the bound its roundings give."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_1903_03837_gb300 import build as B
from test_kernel_radius import CORNERS, POLE, pole_distance, sigma
from test_window_study import F32, lattice_coords, random_queries, window_corner

SOURCE = r"""
#include <cmath>
#include <cuda_runtime.h>
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static inline float __fsqrt_rn(float a) { return std::sqrt(a); }
static inline float __frcp_rn(float a) { return 1.0f / a; }
static inline float __int2float_rn(int a) { return (float)a; }
#include "lf_df.cuh"

extern "C" void z_differences(uint32_t n, int64_t count, const float *qh, const float *ql, const int32_t *b,
                              const int32_t *k, int corners, float *out)
{
    lfk::PointSetK P{};
    P.n = n;
    lfk::fill_z_steps(P);
    for (int64_t q = 0; q < count; ++q) {
        const lfk::ZOffset o = lfk::z_offset(P, b[q], qh[q], ql[q]);
        for (int j = 0; j < corners; ++j) out[q * corners + j] = lfk::z_at(P, o, (float)k[q * corners + j]);
    }
}

extern "C" void chord_lengths(double R, const double O[3], int64_t count, const float *h, const float *d, float *out)
{
    lfk::SphereK S{};
    const double r2 = R * R;
    S.r2_h = (float)r2;
    S.r2_l = (float)(r2 - (double)S.r2_h);
    for (int k = 0; k < 3; ++k) {
        S.o_hi[k] = (float)O[k];
        S.o_lo[k] = (float)(O[k] - (double)S.o_hi[k]);
    }
    for (int64_t i = 0; i < count; ++i)
        out[i] = lfk::chord_length(S, make_float3(h[3 * i], h[3 * i + 1], h[3 * i + 2]),
                                   make_float3(d[3 * i], d[3 * i + 1], d[3 * i + 2]));
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("df")
    src, lib = str(d / "df.cpp"), str(d / "df.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-I", B.CSRC, "-I", B.INCLUDE, "-I", inc,
                    "-o", lib, src], check=True)
    return C.CDLL(lib)


def ptr(a):
    return a.ctypes.data_as(C.c_void_p)


def split(x):
    h = x.astype(np.float32)
    return h, (x - h).astype(np.float32)


@pytest.mark.parametrize("n", [129, 200, 256, 700, 1000, 1500, 3001, 4099, 12288, 16384, 23576, 65536, 100000, 262144,
                               1000003, 1 << 22, 1 << 24])
def test_z_differences_of_the_corners(host, n):
    """q_z - z_i of a lattice window's corners within the radius: two roundings (of
    the difference to the rounded corner, and of the result), the rest far below; and
    in the mean no further off than the differences from the hi/lo point cache."""
    rng = np.random.default_rng(n)
    q = random_queries(rng, 100_000)
    q = q[pole_distance(q, n) >= POLE + 1e-3]
    k, ru, rv, pu, pv = window_corner(lattice_coords(q, n), 0.0, 0.0, 0.0)
    F0, F1 = F32[k], F32[k + 1]
    b = ru * F0 + rv * F1
    G0 = np.where(pu, np.where(pv, F0, -F1), np.where(pv, F1, -F0))
    G1 = np.where(pu, np.where(pv, F1, F0), np.where(pv, -F0, -F1))
    off = np.ascontiguousarray(CORNERS[None, :, 0] * G0[:, None] + CORNERS[None, :, 1] * G1[:, None], np.int32)
    b = np.ascontiguousarray(b, np.int32)
    qh, ql = split(q[:, 2])
    got = np.empty(off.shape, np.float32)
    host.z_differences(C.c_uint32(n), C.c_int64(len(q)), ptr(qh), ptr(ql), ptr(b), ptr(off), len(CORNERS), ptr(got))
    i = b[:, None] + off
    P = oracle.sf_points(n)
    inside = (i >= 0) & (i < n)
    i = np.clip(i, 0, n - 1)
    near = inside & (np.linalg.norm(q[:, None, :] - P[i], axis=2) < sigma(n))
    zi = 1.0 - (2.0 * i + 1.0) / n
    want = q[:, 2:] - zi
    err = np.abs(got - want)
    zb = np.abs(q[:, 2] - (1.0 - (2.0 * b + 1.0) / n))[:, None]
    bound = 2.0 ** -24 * (zb + np.abs(want)) * (1.0 + 2.0 ** -10) + 2.0 ** -29 * sigma(n)
    assert (err <= bound)[near].all(), float((err / bound)[near].max())
    ph, pl = split(zi)
    cached = ((qh[:, None] - ph) + (ql[:, None] - pl)).astype(np.float64)
    rms = np.sqrt(np.mean((err ** 2)[near])), np.sqrt(np.mean(((cached - want) ** 2)[near]))
    assert rms[0] <= 1.02 * rms[1], rms


@pytest.mark.parametrize("R,O", [(1.0, (0.0, 0.0, 0.0)), (2.5, (0.4, -1.2, 0.7)), (0.37, (10.3, 20.1, -7.7)),
                                 (1e-3, (0.0, 1e-3, 0.0)), (150.1, (1.0, 2.0, 3.0))])
def test_chord_lengths(host, R, O):
    """Central to grazing rays, from eyes 1.01 to 40 radii away: one rounding of the
    length, and what 2^-43 of the squares it is formed from makes of it (each
    double-float step is within 2^-46)."""
    rng = np.random.default_rng(int(R * 1000))
    n = 400_000
    O = np.array(O)
    e = random_queries(rng, n) * (R * np.exp(rng.uniform(np.log(1.01), np.log(40.0), n)))[:, None] + O
    # aim at a point of the disc of S seen from the eye, half of them near its rim
    axis = O - e
    u = np.cross(axis, random_queries(rng, n))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    rim = np.where(rng.uniform(size=n) < 0.5, rng.uniform(0, 1, n), 1.0 - 10.0 ** rng.uniform(-5, -1, n))
    L2 = (axis ** 2).sum(1)
    d = axis + u * (rim * R / np.sqrt(L2 - R * R) * np.sqrt(L2))[:, None]
    e32, d32 = e.astype(np.float32), (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    # the front hit, rounded to FP32 as the camera step leaves it
    f = e32.astype(np.float64) - O
    b, c = (f * d32).sum(1), (f * f).sum(1) - R * R
    hits = b * b > c * (d32.astype(np.float64) ** 2).sum(1)
    tn = (-b - np.sqrt(np.maximum(b * b - c, 0.0))).astype(np.float32)
    h = (e32 + (tn[:, None] * d32).astype(np.float32))[hits]
    d32 = np.ascontiguousarray(d32[hits])
    got = np.empty(len(h), np.float32)
    host.chord_lengths(C.c_double(R), ptr(np.ascontiguousarray(O, np.float64)), C.c_int64(len(h)), ptr(h), ptr(d32), ptr(got))
    w = np.longdouble
    f = h.astype(w) - O.astype(w)
    b, c = (f * d32.astype(w)).sum(1), (f * f).sum(1) - w(R) * w(R)
    disc = b * b - c
    inside = disc > 2.0 ** -30 * R * R          # a root whose argument is rounding only says nothing
    assert inside.sum() > 300_000
    root = np.sqrt(disc[inside])
    want = np.maximum(root - b[inside], 0.0)
    size = R * (R + np.abs(O).sum())
    bound = 2.0 ** -24 * (1.0 + 2.0 ** -8) * want + 2.0 ** -43 * (size / root + size / R)
    err = np.abs(got[inside] - want)
    assert (err <= bound).all(), float((err / bound).max())
    assert float(np.median(want)) > 0.1 * R
