"""Texels near the end of FP32's range: a pixel is a weighted mean, so an image of
finite texels is finite, and a texel a ray does not use (the reads of weight 0 in
the blend) does not reach its pixel."""
import numpy as np
import pytest

import lf_inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# 25 taps and the weights' normalisation, a rounding each, with room for a factor of two
RTOL = 64 * 2.0 ** -24


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_03837_gb300 import torch_api
    return torch_api


def views_mix():
    return lf_inputs.pack_offsets([lf_inputs.look_at((2.1, -1.3, 0.8), (0, 0, 0), 93, 61),
                                   lf_inputs.look_at((0.05, 0.02, 2.4), (0, 0, 0), 48, 48),
                                   lf_inputs.look_at((1.9, 0.4, 0.0), (0, 0, 0.2), 64, 33)])


@pytest.mark.parametrize("upper", [False, True])
@pytest.mark.parametrize("K", [5, 9, 1])
@pytest.mark.parametrize("dtype,C", [("f32", 4), ("f32", 3), ("f16", 4), ("e4m3", 4)])
def test_constant_table_at_the_end_of_the_range(api, dtype, C, K, upper):
    """A table of 3.3e38 renders 3.3e38."""
    M, N, top = 700, 300, 3.3e38
    rows = M // 2 if upper else M
    T = torch.full((rows, N, C), top, device="cuda")
    codes, scales = (T, None) if dtype == "f32" else api.quantize_table(T, dtype)
    lf = api.LightField(codes, dtype, scales, n_origins=M, upper=upper, k_nearest=K)
    for with_idx in (False, True):
        out, _ = lf.render(views_mix(), with_idx=with_idx)
        hit = out[:, 0] != 0
        assert int(hit.sum()) > 1000
        assert torch.isfinite(out).all()
        assert float((out[hit].double() / float(np.float32(top)) - 1.0).abs().max()) <= RTOL
    lf.sync_status()
    lf.close()


@pytest.mark.parametrize("K", [5, 9])
@pytest.mark.parametrize("dtype,C", [("f32", 4), ("f32", 3), ("e4m3", 4)])
def test_large_texels_of_the_first_row_stay_with_their_rays(api, dtype, C, K):
    """Row 0 holds 3.3e38, the others values up to 1: rays without origin 0 have the
    same pixels as with an ordinary row 0."""
    M, N = 700, 300
    T = torch.from_numpy(np.random.default_rng(4).uniform(0.1, 1, (M, N, C)).astype(np.float32)).cuda()
    big = T.clone()
    big[0] = 3.3e38
    outs = []
    for t in (T, big):
        codes, scales = (t, None) if dtype == "f32" else api.quantize_table(t, dtype)
        lf = api.LightField(codes, dtype, scales, k_nearest=K)
        outs.append(lf.render(views_mix())[0])
        idx = lf.render(views_mix(), with_idx=True)[1]
        lf.sync_status()
        lf.close()
    without = (idx[:, :K] != 0).all(1)
    assert 0 < int((~without).sum()) < int((idx[:, 0] >= 0).sum())
    assert torch.equal(outs[0][without], outs[1][without])
    assert torch.isfinite(outs[1]).all()
