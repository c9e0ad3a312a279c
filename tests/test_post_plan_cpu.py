"""The post-filter's chunk length (csrc/lf_post_plan.h) against a search over every
length: the fewest steps by the plan's own cost, ceil(CTAs / slots) waves of (bands +
2.3) steps, also where the strips alone exceed the resident slots."""
import ctypes as C
import math
import shutil
import subprocess

import pytest

from paper_1903_03837_gb300 import build as B

SOURCE = r"""
#include "lf_post_plan.h"
extern "C" uint64_t chunk_bands(const uint64_t *strips, const uint64_t *bands, uint32_t n, uint64_t slots)
{
    lfk::PostExtent v[32];
    for (uint32_t k = 0; k < n; ++k) v[k] = {strips[k], bands[k]};
    return lfk::post_chunk_bands(v, n, slots);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("plan")
    src, lib = str(d / "plan.cpp"), str(d / "plan.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O2", "-shared", "-fPIC", "-I", B.CSRC, "-o", lib, src], check=True)
    L = C.CDLL(lib)
    L.chunk_bands.restype = C.c_uint64

    def chunk(sizes, slots):
        s = (C.c_uint64 * len(sizes))(*[(w + 123) // 124 for w, _ in sizes])
        b = (C.c_uint64 * len(sizes))(*[(h + 5) // 6 for _, h in sizes])
        return int(L.chunk_bands(s, b, len(sizes), C.c_uint64(slots)))
    return chunk


@pytest.mark.parametrize("sizes", [
    [(1920, 1080)], [(1, 1)], [(256, 256)], [(3840, 2160)] * 2, [(1440, 1600)] * 2, [(640, 480), (37, 1021), (2048, 3)],
    [(1920, 1080)] * 20, [(1240, 302)] * 32, [(1440, 1600)] * 26, [(1440, 1600)] * 32, [(65536, 40)], [(65536, 1)] * 32,
    [(65536, 65536)], [(1, 1080)] * 32, [(124, 7)] * 31 + [(3840, 2160)]])
@pytest.mark.parametrize("slots", [304, 152, 7])
def test_chunk_length_takes_the_fewest_steps(plan, sizes, slots):
    strips, bands = [(w + 123) // 124 for w, _ in sizes], [(h + 5) // 6 for _, h in sizes]

    def waves(n):
        return math.ceil(sum(s * ((b + n - 1) // n) for s, b in zip(strips, bands)) / slots)
    least = waves(max(bands))
    chosen = plan(sizes, slots)
    assert 1 <= chosen <= max(bands)
    best = min(waves(n) * (n + 2.3) for n in range(1, max(bands) + 1) if waves(n) <= least + 3)
    assert waves(chosen) * (chosen + 2.3) == pytest.approx(best, rel=1e-12)
