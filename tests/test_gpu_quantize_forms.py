"""The per-row quantiser over the forms its launch chooses by: rows held by a warp,
by a CTA, read twice; RGB rows that are whole groups of four texels and not; source
buffers off a 16-byte boundary; values at the codes' rounding ties, zeros of either
sign, denormals, rows whose scale is denormal, tiny or huge. Codes and scales equal
the oracle's, byte for byte."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_03837_gb300 import torch_api
    return torch_api


def table(M, N, C, dtype, seed):
    rng = np.random.default_rng(seed)
    T = (rng.standard_normal((M, N, C)) * 10.0 ** rng.uniform(-4, 4, (M, 1, 1))).astype(np.float32)
    # every third row: values at and next to the midpoints of neighbouring codes times the row's scale
    top = 448.0 if dtype == "e4m3" else 1.0
    for i in range(0, M, 3):
        amax = np.float32(10.0 ** rng.uniform(-3, 3))
        s = np.float32(amax / np.float32(448.0)) if dtype == "e4m3" else amax
        mant = rng.integers(0, 16 if dtype == "e4m3" else 4096, (N, C)) + 0.5
        e = rng.integers(-12, 5 if dtype == "e4m3" else -10, (N, C))
        v = np.ldexp(mant, e) * float(s)
        v = np.minimum(v, top * float(s)).astype(np.float32)
        step = rng.integers(-1, 2, (N, C))
        v = np.where(step > 0, np.nextafter(v, np.float32(np.inf)), np.where(step < 0, np.nextafter(v, np.float32(0)), v))
        T[i] = np.where(rng.random((N, C)) < 0.5, -v, v)
        T[i, 0, 0] = amax
    if M > 7:
        T[1] = 0
        T[2, :, 0] = -0.0
        T[4] *= np.float32(1e-30)
        T[5] = (T[5] / np.abs(T[5]).max() * np.float32(1e-39)).astype(np.float32)      # a denormal scale
        T[7] = T[7] / np.abs(T[7]).max() * np.float32(3e38)
        T[7, -1, -1] = np.float32(-1e-42)
    return T


@pytest.mark.parametrize("dtype", ["f16", "e4m3"])
@pytest.mark.parametrize("C", [3, 4])
@pytest.mark.parametrize("N", [1, 4, 63, 64, 65, 128, 129, 256, 260, 512, 1000, 1024, 2050, 4096, 4100])
def test_codes_and_scales_are_the_oracles(api, N, C, dtype):
    T = table(13, N, C, dtype, N * 8 + C)
    want, want_s = oracle.quantize_rows(T, dtype)
    for off in (0, 1, 2):
        buf = torch.zeros(T.size + 4, device="cuda")
        src = buf[off:off + T.size].view(T.shape)
        src.copy_(torch.from_numpy(T))
        codes, s = api.quantize_table(src, dtype)
        np.testing.assert_array_equal(s.cpu().numpy(), want_s)
        got = codes.cpu().numpy()
        got = got.view(np.uint16) if dtype == "f16" else got
        np.testing.assert_array_equal(got[..., :C], want)
        assert np.all(got[..., C:] == 0)


@pytest.mark.parametrize("dtype", ["f16", "e4m3"])
def test_the_division_is_correctly_rounded(api, dtype):
    """Rows of one scale each, 16,384 values: codes equal those of NumPy's FP32
    quotient."""
    rng = np.random.default_rng(3)
    T = rng.uniform(-1, 1, (64, 4096, 4)).astype(np.float32) * np.float32(2) ** rng.integers(-20, 20, (64, 1, 1)).astype(np.float32)
    want, want_s = oracle.quantize_rows(T, dtype)
    codes, s = api.quantize_table(torch.from_numpy(T).cuda(), dtype)
    got = codes.cpu().numpy()
    np.testing.assert_array_equal(s.cpu().numpy(), want_s)
    np.testing.assert_array_equal(got.view(np.uint16) if dtype == "f16" else got, want)
