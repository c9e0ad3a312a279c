"""The backward scatter over the forms its warp sums take: warps that share a few
neighbours (matrix sums), warps of scattered rays (tap by tap), gradients that
are not finite, 3 and 4 channels, 5, 9 and nearest sampling, upper-hemisphere
tables, and the same from the forward's indices. Against the oracle's adjoint."""
import numpy as np
import pytest

import lf_inputs
import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_03837_gb300 import torch_api
    return torch_api


def views_mix():
    return lf_inputs.pack_offsets([lf_inputs.look_at((2.1, -1.3, 0.8), (0, 0, 0), 96, 72, fov_y_deg=6.0),   # close: shared
                                   lf_inputs.look_at((2.4, 0.6, -0.7), (0, 0, 0), 45, 31),                  # scattered
                                   lf_inputs.look_at((0.05, 0.02, 2.4), (0, 0, 0), 40, 40, fov_y_deg=20.0),
                                   lf_inputs.look_at((1.9, 0.4, 0.0), (0, 0, 0.2), 64, 33)])


@pytest.mark.parametrize("upper", [False, True])
@pytest.mark.parametrize("K", [5, 9, 1])
@pytest.mark.parametrize("M,N,C", [(60, 45, 4), (1024, 256, 3), (3001, 700, 4), (5, 3, 3)])
def test_backward_against_the_oracle(api, M, N, C, K, upper):
    rows = M // 2 if upper else M
    rng = np.random.default_rng(M + C + K)
    T = rng.uniform(0, 1, (rows, N, C)).astype(np.float32)
    views = views_mix()
    P = lf_inputs.total_pixels(views)
    g = rng.standard_normal((P, C)).astype(np.float32)
    pix = lf_inputs.pixel_list(views)
    offs = lf_inputs.pixel_offsets(views, pix)
    want = oracle.render_backward(oracle.Scene(M, N, C, "f32", T, K=K, upper=upper), views, pix, g[offs].astype(np.float64))
    lf = api.LightField(torch.from_numpy(T).cuda(), "f32", n_origins=M, upper=upper, k_nearest=K)
    _, idx = lf.render(views, with_idx=True)
    gd = torch.from_numpy(g).cuda()
    tol = 2e-5 * max(1.0, np.abs(want).max())           # FP32 atomics in any order, as the other backward tests
    for given in (None, idx):
        got = lf.render_backward(views, gd, idx=given).cpu().numpy().astype(np.float64)
        lf.sync_status()
        assert np.abs(got - want).max() <= tol, given is None
    lf.close()


def test_gradients_that_are_not_finite_stay_with_their_texels(api):
    """An infinite or NaN image gradient reaches the texels its own ray blends and
    no others."""
    M, N, C = 1024, 256, 3
    T = np.random.default_rng(1).uniform(0, 1, (M, N, C)).astype(np.float32)
    views = views_mix()[:1]
    P = lf_inputs.total_pixels(views)
    lf = api.LightField(torch.from_numpy(T).cuda(), "f32")
    g = torch.ones((P, C), device="cuda")
    clean = lf.render_backward(views, g)
    hot = P // 2 + 7
    only = torch.zeros_like(g)
    only[hot] = 1.0
    touched = lf.render_backward(views, only)[..., 0] != 0
    assert 1 <= int(touched.sum()) <= 25
    for bad in (float("inf"), float("-inf"), float("nan")):
        g2 = g.clone()
        g2[hot] = bad
        got = lf.render_backward(views, g2)
        assert torch.equal(~torch.isfinite(got[..., 0]), touched)
        keep = ~touched
        assert torch.allclose(got[keep], clean[keep], rtol=1e-4, atol=1e-6)
    lf.sync_status()
    lf.close()


def test_autograd_gradient_is_the_backward(api):
    """RenderFunction's gradient equals render_backward's (nearest sampling too)."""
    M, N, C = 512, 130, 4
    views = views_mix()
    for K in (5, 1, 9):
        T = torch.rand((M, N, C), device="cuda").requires_grad_(True)
        lf = api.LightField(T.detach(), "f32", borrow=True, k_nearest=K)
        g = torch.randn((lf_inputs.total_pixels(views), C), device="cuda")
        img = api.render(T, lf, views)
        got, = torch.autograd.grad(img, T, grad_outputs=g)
        want = lf.render_backward(views, g)
        assert torch.allclose(got, want, rtol=1e-4, atol=1e-4)
        lf.close()
