"""A kernel launch that fails reports its error to the caller and leaves none behind
for the next launch to report. The library's objects are linked with stand-ins for
the runtime's launch and last-error calls, so no GPU is needed."""
import glob
import os
import subprocess

from paper_1903_03837_gb300 import build as B

SOURCE = r"""
#include <cstdio>
#include <cstring>
#include <cuda_runtime.h>
#include "lf_kernels.h"

static cudaError_t last = cudaSuccess;
extern "C" {
cudaError_t __wrap_cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t)
{
    return last = cudaErrorInvalidConfiguration;
}
cudaError_t __wrap_cudaGetLastError()
{
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
cudaError_t __wrap_cudaGetDevice(int *dev) { *dev = 0; return cudaSuccess; }
cudaError_t __wrap_cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 4; return cudaSuccess; }
cudaError_t __wrap_cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *, const void *, int, size_t)
{
    return last = cudaErrorInvalidDeviceFunction;
}
}

static int bad = 0;
static void expect(const char *what, cudaError_t e)
{
    if (e == cudaErrorInvalidConfiguration && last == cudaSuccess) return;
    printf("%s: returned %d, left %d\n", what, (int)e, (int)last);
    last = cudaSuccess;
    ++bad;
}

template <int MAXV>
static void renders()
{
    static lfk::RenderParams<MAXV> p;
    memset(&p, 0, sizeof p);
    expect("render", lfk::launch_render(lfk::kF32C4, p, dim3(1), 256, nullptr));
    expect("backward", lfk::launch_backward(p, dim3(1), 256, nullptr));
    expect("fixup", lfk::launch_fixup(lfk::kF32C4, false, p, nullptr));
    expect("backward fixup", lfk::launch_fixup(lfk::kF32C4, true, p, nullptr));
}

int main()
{
    renders<lfk::kSmallViews>();
    renders<lfk::kLargeViews>();
    static lfk::PrecomputeParams q;
    memset(&q, 0, sizeof q);
    q.rows = q.N = 1;
    expect("precompute", lfk::launch_precompute(q, nullptr));
    lf_view v{};
    v.eye[0] = 3.0f;
    v.forward[0] = -1.0f;
    v.width = v.height = 16;
    const double O[3] = {0.0, 0.0, 0.0};
    lfk::SphereK S{};
    lf_view vs[3] = {v, v, v};
    expect("volume, one view", lfk::launch_volume_direct(q, vs, 1, S, 1.0, O, nullptr));
    expect("volume, three views", lfk::launch_volume_direct(q, vs, 3, S, 1.0, O, nullptr));
    if (!bad) printf("ok\n");
    return bad;
}
"""
WRAPPED = ("cudaLaunchKernel", "cudaGetLastError", "cudaGetDevice", "cudaDeviceGetAttribute",
           "cudaOccupancyMaxActiveBlocksPerMultiprocessor")


def test_a_failed_launch_leaves_no_error_behind(tmp_path):
    B.build(force=not glob.glob(os.path.join(B.BUILD, "lf_*.o")))
    src, exe = str(tmp_path / "launch_errors.cu"), str(tmp_path / "launch_errors")
    with open(src, "w") as f:
        f.write(SOURCE)
    objs = sorted(glob.glob(os.path.join(B.BUILD, "lf_*.o")))
    wrap = [a for w in WRAPPED for a in ("-Xlinker", f"--wrap={w}")]
    r = subprocess.run([B.nvcc(), *B.ARCH, "-std=c++17", "-I", B.INCLUDE, "-I", B.CSRC, *wrap, "-o", exe, src, *objs],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
