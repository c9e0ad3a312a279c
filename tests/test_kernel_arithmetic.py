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
