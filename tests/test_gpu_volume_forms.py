"""The precompute and the direct volume render over the forms their kernels
branch on: every number of blob pairs (0 to 16 blobs), steps dense enough to pass
the polynomial's range (optical depth of a step above 1) and so dense that nothing
is left behind them, views that fill tiles partly, more views than one launch
holds, a moved and scaled sphere. Tolerance as in test_gpu_precompute."""
import numpy as np
import pytest

import lf_inputs
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_03837_gb300 import torch_api
    return torch_api


def tol(vol, want):
    return 1e-5 + vol.steps * 2.0 ** -21 * (1.0 + np.abs(want))


@pytest.mark.parametrize("B", [0, 1, 2, 3, 5, 6, 7, 8, 9, 11, 13, 15, 16])
def test_every_number_of_blobs(api, B):
    vol = lf_inputs.draw_volume(B + 1, B=B, spp=2, steps=12)
    got = api.precompute_table(vol, 130, 37, 4).cpu().numpy()
    want = oracle.volume_table(vol, 130, 37, 4)
    assert (np.abs(got - want) <= tol(vol, want)).all()
    views = lf_inputs.pack_offsets([lf_inputs.look_at((2.2, -1.1, 0.9), (0, 0, 0), 37, 21)])
    got = api.render_volume(vol, views, 4).cpu().numpy()
    want, hits = oracle.volume_pixels(vol, views, lf_inputs.pixel_list(views))
    assert hits > 50 and (np.abs(got - want) <= tol(vol, want)).all()


@pytest.mark.parametrize("steps,scale", [(1, 1.0), (2, 4.0), (8, 30.0), (64, 200.0)])
def test_dense_steps(api, steps, scale):
    """Optical depths of a step from below 1/16 to some hundreds."""
    vol = lf_inputs.draw_volume(3, B=8, spp=2, steps=steps)
    vol.dens = np.ascontiguousarray((vol.dens * scale).astype(np.float32).astype(np.float64))
    got = api.precompute_table(vol, 200, 64, 4).cpu().numpy()
    want = oracle.volume_table(vol, 200, 64, 4)
    # the 1e-5 for the ray geometry is per density up to 12 / R
    assert (np.abs(got - want) <= 1e-5 * scale + steps * 2.0 ** -21 * (1.0 + np.abs(want))).all()


@pytest.mark.parametrize("C", [3, 4])
def test_many_uneven_views_of_a_moved_sphere(api, C):
    """70 views (launches of 32, 32 and 6), sizes around the 16-pixel tiles."""
    vol = lf_inputs.draw_volume(9, B=5, R=2.5, O=(0.4, -1.2, 0.7), spp=1, steps=9)
    rng = np.random.default_rng(2)
    vs = []
    for k in range(70):
        d = rng.normal(size=3)
        d *= 2.5 * rng.uniform(1.2, 3.0) / np.linalg.norm(d)
        c = np.array([0.4, -1.2, 0.7])
        vs.append(lf_inputs.look_at(tuple(c + d), tuple(c + 0.3 * rng.normal(size=3)), int(rng.choice([1, 7, 15, 16, 17, 33])),
                                    int(rng.choice([1, 5, 16, 18, 31]))))
    views = lf_inputs.pack_offsets(vs)
    got = api.render_volume(vol, views, C).cpu().numpy()
    want, hits = oracle.volume_pixels(vol, views, lf_inputs.pixel_list(views))
    assert hits > 1000
    assert (np.abs(got - want[:, :C]) <= tol(vol, want[:, :C])).all()


def test_grazing_rays_of_a_distant_eye(api):
    """Chords from grazing to central, seen from 30 radii: the opacity of a nearly
    uniform medium follows the chord's length."""
    vol = lf_inputs.draw_volume(4, B=1, spp=1, steps=4)
    vol.width[:] = 4.0
    vol.dens[:] = 1.0
    views = lf_inputs.pack_offsets([lf_inputs.look_at((30.0, 3.0, -2.0), (0, 0, 0), 64, 64, fov_y_deg=4.0)])
    got = api.render_volume(vol, views, 4).cpu().numpy()
    want, hits = oracle.volume_pixels(vol, views, lf_inputs.pixel_list(views))
    assert hits > 500 and (np.abs(got - want) <= tol(vol, want)).all()
