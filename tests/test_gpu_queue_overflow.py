"""More uncertain rays in one launch than the queue of the exact pass holds (2^18, or
LF_NOALLOC_MAX_DEFERRED without allocation): the exact pass then takes every ray
of the launch, and in the backward tells the rays that are scattered already from
the others by searching again.

A view whose image plane has no extent sends the same ray through every pixel.
That ray is aimed at a near-tie the FP32 distances cannot order: for indices, two
of the 6 nearest origins at the same distance; for an upper-hemisphere table
(images and gradients), a ray past the rim with no stored origin within the
kernel radius and another point as far as the nearest stored one. A second,
ordinary view of the same launch has rays that settle."""
import ctypes as C

import numpy as np
import pytest

import lf_inputs
import oracle
from paper_1903_03837_gb300 import lumipath as lp
from test_gpu_adversarial import _unit, chord_views, cKDTree, tie_targets

torch = pytest.importorskip("torch")

QUEUE = 1 << 18
ATOL = 1e-5


def all_one_ray(view, side):
    return lf_inputs.View(view.eye, view.right, view.up, view.forward, 0.0, 0.0, side, side, 0)


def ordinary():
    return lf_inputs.look_at((2.1, -1.3, 0.8), (0, 0, 0), 61, 47)


def origin_tie_view(M):
    """A 1x1 view whose front hit ties the r-th and (r+1)-th nearest origins, r <= 5,
    within 2^-22 of their squared distance: the keys of the ranking, with 4 bits of it
    dropped, are equal or neighbours."""
    rng = np.random.default_rng(11)
    P = oracle.sf_points(M)
    t, _ = tie_targets(P, cKDTree(P), rng, 400, 5)
    for v in chord_views(t, _unit(rng.standard_normal((len(t), 3))), rng):
        hit, _, _, _, qo, _ = oracle.trace_pixel(1.0, (0.0, 0.0, 0.0), v, 0, 0)
        d2 = np.sort(((P - qo) ** 2).sum(1))[:6]
        if hit and (np.diff(d2) < 2.0 ** -22 * d2[1:]).any():
            return v
    raise AssertionError("no tie found")


def rim_tie_view(M):
    """A 1x1 view whose front hit has no stored origin (rows below M/2) within the
    kernel radius, the nearest stored one among the 4 nearest origins, and another
    point as far as that one within half the kernel's FP32 bound (2^-16 of the squared
    radius)."""
    rng = np.random.default_rng(12)
    P, rows, s2 = oracle.sf_points(M), M // 2, 4.0 * np.pi / M
    for _ in range(200000):
        q = _unit(rng.standard_normal(3))
        q[2] = -abs(q[2]) * rng.uniform(0, 1)
        q = _unit(q)
        d2 = ((P - q) ** 2).sum(1)
        near = np.argsort(d2)[:4]
        stored = near[near < rows]
        if len(stored) == 0 or stored[0] == near[0]:
            continue
        s, u = stored[0], near[list(near).index(stored[0]) - 1]
        w = P[u] - P[s]
        q = _unit(q - (q @ w) / (w @ w) * w)
        v = chord_views(q[None], _unit(rng.standard_normal((1, 3))), rng)[0]
        hit, _, _, _, qo, _ = oracle.trace_pixel(1.0, (0.0, 0.0, 0.0), v, 0, 0)
        d2 = ((P - qo) ** 2).sum(1)
        near = np.argsort(d2)
        if hit and d2[:rows].min() > s2 * 1.001 and s in near[:4] and np.argmin(d2[:rows]) == s and \
                abs(d2[u] - d2[s]) < 2.0 ** -17 * s2 and qo[2] > -1.7 * s2 ** 0.5:
            return v
    raise AssertionError("no tie at the rim found")


def test_the_tie_views_exist():
    origin_tie_view(3001)
    rim_tie_view(64)


@pytest.fixture(scope="module")
def api():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_03837_gb300 import torch_api
    return torch_api


def views_of(tie, side):
    return lf_inputs.pack_offsets([all_one_ray(tie, side), ordinary()])


@pytest.mark.gpu
def test_indices_when_the_queue_overflows(api):
    M, N, side = 3001, 257, 520
    tie = origin_tie_view(M)
    assert side * side > QUEUE
    T = np.random.default_rng(1).uniform(0, 1, (M, N, 4)).astype(np.float32)
    scene = oracle.Scene(M, N, 4, "f32", T)
    want1, idx1, _ = oracle.render_views(scene, lf_inputs.pack_offsets([tie]))
    want2, idx2, _ = oracle.render_views(scene, lf_inputs.pack_offsets([ordinary()]))
    lf = api.LightField(torch.from_numpy(T).cuda(), "f32")
    for views in (views_of(tie, side), views_of(tie, 8), views_of(tie, side)):   # the queue is reset in between
        out, idx = lf.render(views, with_idx=True)
        lf.sync_status()
        out, idx = out.cpu().numpy(), idx.cpu().numpy()
        n = views[1].out_offset
        assert (idx[:n] == idx1[0]).all() and np.array_equal(idx[n:], idx2)
        assert np.abs(out[:n] - want1[0]).max() <= ATOL and np.abs(out[n:] - want2).max() <= ATOL
    lf.close()


@pytest.mark.gpu
def test_indices_without_allocation_when_the_queue_overflows(api):
    M, N, side = 3001, 257, 130
    tie = origin_tie_view(M)
    T = np.random.default_rng(1).uniform(0, 1, (M, N, 4)).astype(np.float32)
    scene = oracle.Scene(M, N, 4, "f32", T)
    want1, idx1, _ = oracle.render_views(scene, lf_inputs.pack_offsets([tie]))
    want2, idx2, _ = oracle.render_views(scene, lf_inputs.pack_offsets([ordinary()]))
    d = lp.lf_table_desc()
    d.radius = 1.0
    d.n_origins, d.n_directions, d.channels, d.k_nearest = M, N, 4, 5
    d.dtype = lp.DTYPES["f32"]
    Td = torch.from_numpy(T).cuda()
    st = torch.cuda.current_stream().cuda_stream
    for views in (views_of(tie, side), views_of(tie, 8)):
        n = views[1].out_offset
        P = lf_inputs.total_pixels(views)
        assert side * side > 16384
        out = torch.empty((P, 4), device="cuda")
        idx = torch.empty((P, 10), dtype=torch.int32, device="cuda")
        lp._check(lp.lib().lf_render_noalloc(C.byref(d), C.c_void_p(Td.data_ptr()), None, lp.make_views(views), 2, None,
                                             C.c_void_p(out.data_ptr()), C.c_void_p(idx.data_ptr()), C.c_void_p(st or None)))
        lp._check(lp.lib().lf_noalloc_sync_status(C.c_void_p(st or None)))
        out, idx = out.cpu().numpy(), idx.cpu().numpy()
        assert (idx[:n] == idx1[0]).all() and np.array_equal(idx[n:], idx2)
        assert np.abs(out[:n] - want1[0]).max() <= ATOL and np.abs(out[n:] - want2).max() <= ATOL


@pytest.mark.gpu
@pytest.mark.parametrize("K", [5, 1])
def test_upper_hemisphere_image_and_gradient_when_the_queue_overflows(api, K):
    """With K = 1 no ray of this kind is queued (the nearest origin alone counts):
    the same answers without an overflow."""
    M, N, side = 64, 33, 520
    rows = M // 2
    tie = rim_tie_view(M)
    rng = np.random.default_rng(2)
    T = rng.uniform(0.1, 1, (rows, N, 4)).astype(np.float32)
    scene = oracle.Scene(M, N, 4, "f32", T, K=K, upper=True)
    want1, _, _ = oracle.render_views(scene, lf_inputs.pack_offsets([tie]))
    want2, _, _ = oracle.render_views(scene, lf_inputs.pack_offsets([ordinary()]))
    lf = api.LightField(torch.from_numpy(T).cuda(), "f32", n_origins=M, upper=True, k_nearest=K)
    views = views_of(tie, side)
    n, P = views[1].out_offset, lf_inputs.total_pixels(views)
    for _ in range(2):
        out = lf.render(views)[0].cpu().numpy()
        lf.sync_status()
        assert np.abs(out[:n] - want1[0]).max() <= ATOL and np.abs(out[n:] - want2).max() <= ATOL
    if K == 5:
        assert np.abs(want1).max() > 0
    # gradients of 200 pixels of the first view, the last ones (past the queue's end
    # when it fills in order) among them, and of all of the second
    some = np.unique(np.concatenate([rng.integers(0, n, 180), np.arange(n - 20, n)]))
    g = np.zeros((P, 4), np.float32)
    g[some] = rng.standard_normal((len(some), 4))
    g[n:] = rng.standard_normal((P - n, 4))
    one = lf_inputs.pack_offsets([tie])
    want = oracle.render_backward(scene, one, lf_inputs.pixel_list(one), g[some].astype(np.float64).sum(0, keepdims=True))
    two = lf_inputs.pack_offsets([ordinary()])
    want = want + oracle.render_backward(scene, two, lf_inputs.pixel_list(two), g[n:].astype(np.float64))
    tol = 2e-5 * max(1.0, np.abs(want).max())
    for _ in range(2):
        got = lf.render_backward(views, torch.from_numpy(g).cuda()).cpu().numpy().astype(np.float64)
        lf.sync_status()
        assert np.abs(got - want).max() <= tol
    lf.close()
