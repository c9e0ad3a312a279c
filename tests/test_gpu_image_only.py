"""Images without an index output: the render lists the points within the filter
kernel's radius instead of ranking the nearest ones (5 or 9 neighbours), or
takes the nearest listed one (nearest sampling). The same views with an index
output go through the ranking, and store the same image: every storage form,
neighbour count, table with all rows or the upper hemisphere's, sizes from the
full scan through the poles to windows, image type and launch shape. Against the
oracle: colours within 1e-5 for FP32 tables (as the other render tests)."""
import numpy as np
import pytest

import lf_inputs
import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ATOL = 1e-5


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_03837_gb300 import torch_api
    return torch_api


def views_mix():
    return lf_inputs.pack_offsets([lf_inputs.look_at((2.1, -1.3, 0.8), (0, 0, 0), 93, 61),
                                   lf_inputs.look_at((0.05, 0.02, 2.4), (0, 0, 0), 48, 48),        # over a pole
                                   lf_inputs.look_at((0.1, -0.05, -2.2), (0.1, 0.1, 0), 40, 37),   # under the other
                                   lf_inputs.look_at((1.9, 0.4, 0.0), (0, 0, 0.2), 64, 33),        # across the rim
                                   lf_inputs.look_at((0.3, 0.2, 0.1), (0, 0, 0), 32, 32),          # eye inside S
                                   lf_inputs.look_at((6.0, 4.0, 1.0), (6.0, 4.0, 3.0), 35, 20)])   # S behind or beside


@pytest.mark.parametrize("upper", [False, True])
@pytest.mark.parametrize("K", [5, 9, 1])
@pytest.mark.parametrize("M,N", [(2, 1), (7, 5), (100, 60), (129, 131), (1024, 256), (3001, 700)])
def test_image_without_indices_f32(api, M, N, K, upper):
    rows = M // 2 if upper else M
    T = np.random.default_rng(M + K).uniform(0, 1, (rows, N, 4)).astype(np.float32)
    views = views_mix()
    want, _, hits = oracle.render_views(oracle.Scene(M, N, 4, "f32", T, K=K, upper=upper), views)
    assert hits > 0
    lf = api.LightField(torch.from_numpy(T).cuda(), "f32", n_origins=M, upper=upper, k_nearest=K)
    for launch in ({}, dict(tile_w=8, tile_h=16, warp_w=4, order=1, persistent=1)):
        lf.set_launch(**launch)
        alone, _ = lf.render(views)
        both, idx = lf.render(views, with_idx=True)
        lf.sync_status()
        assert np.abs(alone.cpu().numpy() - want).max() <= ATOL
        assert torch.equal(alone, both)
        assert torch.equal(alone.abs().sum(1) > 0, idx[:, 0] >= 0)
    lf.close()


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("K", [5, 1])
@pytest.mark.parametrize("dtype,C", [("f32", 3), ("f16", 4), ("e4m3", 4)])
def test_image_without_indices_storage_forms(api, dtype, C, K, half):
    M, N = 4099, 515
    T = torch.from_numpy(np.random.default_rng(C).uniform(0, 2, (M, N, C)).astype(np.float32)).cuda()
    codes, scales = (T, None) if dtype == "f32" else api.quantize_table(T, dtype)
    lf = api.LightField(codes, dtype, scales, R=1.7, O=(0.2, -0.1, 0.4), k_nearest=K)
    views = views_mix()
    alone, _ = lf.render(views, half=half)
    both, _ = lf.render(views, with_idx=True, half=half)
    lf.sync_status()
    assert (alone != 0).any()
    assert torch.equal(alone, both)
    lf.close()


def test_table_beyond_four_gib(api):
    """A table of more than 4 GiB takes 64-bit texel offsets: the same image as
    the first rows of it hold in a smaller table."""
    M, N = 70001, 1024
    big = torch.zeros((M, 4 * N, 4), device="cuda")          # 4.27 GiB
    g = torch.Generator(device="cuda").manual_seed(3)
    rowv = torch.rand((M, 1, 4), generator=g, device="cuda")
    big += rowv                                              # constant along each origin row
    small = rowv.expand(M, N, 4).contiguous()
    views = views_mix()
    lf = api.LightField(big, "f32", borrow=True)
    a, _ = lf.render(views)
    lf.close()
    lf = api.LightField(small, "f32", borrow=True)
    b, _ = lf.render(views)
    lf.close()
    assert (a != 0).any()
    assert float((a - b).abs().max()) <= ATOL


def test_screen_bound_keeps_every_hit(api):
    """Cameras at many distances, some with a basis that is neither orthogonal
    nor of unit length: the pixels the library hits are the oracle's (an image of
    a constant table is the constant exactly where the ray hits)."""
    rng = np.random.default_rng(8)
    vs = []
    for k in range(24):
        d = rng.normal(size=3)
        d *= rng.choice([1.05, 1.5, 3.0, 9.0, 40.0]) / np.linalg.norm(d)
        v = lf_inputs.look_at(tuple(d), tuple(0.7 * rng.normal(size=3)), int(rng.integers(17, 90)), int(rng.integers(17, 90)),
                              fov_y_deg=float(rng.uniform(3, 100)))
        if k % 3 == 0:
            r = np.array(v.right) * 1.3 + 0.2 * np.array(v.up)
            u = np.array(v.up) * 0.8 - 0.1 * np.array(v.forward)
            v = lf_inputs.View(v.eye, tuple(float(np.float32(x)) for x in r), tuple(float(np.float32(x)) for x in u),
                               v.forward, v.tan_half_x, v.tan_half_y, v.width, v.height, 0)
        vs.append(v)
    views = lf_inputs.pack_offsets(vs)
    T = np.ones((64, 32, 4), np.float32)
    _, want_idx, hits = oracle.render_views(oracle.Scene(64, 32, 4, "f32", T), views)
    lf = api.LightField(torch.from_numpy(T).cuda(), "f32")
    for tile in (dict(tile_w=16, tile_h=16, warp_w=8), dict(tile_w=8, tile_h=4, warp_w=8)):
        lf.set_launch(**tile)
        out, _ = lf.render(views)
        assert hits > 100
        assert np.array_equal(out.cpu().numpy()[:, 0] > 0, want_idx[:, 0] >= 0)
    lf.close()
