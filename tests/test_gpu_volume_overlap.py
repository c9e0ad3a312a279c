"""Views of a direct volume render that overlap in the output: the last one stays, as
if each had its own launch (disjoint views share one)."""
import numpy as np
import pytest

import lf_inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C", [3, 4])
@pytest.mark.parametrize("offsets", [(0, 0), (0, 500), (0, 961, 500, 1922), (40, 0, 1500, 1001, 3000, 2039, 0)])
def test_the_last_of_overlapping_views_stays(offsets, C):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_03837_gb300 import torch_api as api
    vol = lf_inputs.draw_volume(5, B=4, spp=1, steps=9)
    views = []
    for k, off in enumerate(offsets):
        v = lf_inputs.look_at((2.2 + 0.1 * k, -1.1, 0.3 * k), (0, 0, 0), 31, 31)
        views.append(lf_inputs.View(v.eye, v.right, v.up, v.forward, v.tan_half_x, v.tan_half_y, 31, 31, off))
    P = lf_inputs.total_pixels(views)
    want = torch.full((P, C), -1.0, device="cuda")
    for v in views:
        api.render_volume(vol, [v], C, out=want)
    for _ in range(5):
        got = torch.full((P, C), -1.0, device="cuda")
        api.render_volume(vol, views, C, out=got)
        # the kernels of one, two and more views round alike up to contraction
        assert float((got - want).abs().max()) <= 1e-5
    assert int((want > 0).sum()) > 100 and np.isfinite(want.cpu().numpy()).all()
