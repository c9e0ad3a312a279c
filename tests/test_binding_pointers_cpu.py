"""The binding takes device addresses as integers (or None): the host address of a
bytes object, a string, an array or another pointer is refused, not passed on to a
kernel. Every call here has another argument that the library refuses, so nothing is
launched if one slips through."""
import ctypes as C

import pytest

from paper_1903_03837_gb300 import lumipath as lp

NOT_ADDRESSES = [b"0123456789abcdef", "text", (C.c_float * 4)(), C.c_void_p(64), C.c_char_p(b"x"), 1.5]
A = 1 << 20


def calls(x):
    views = lp.make_views([])
    d = lp.lf_precompute_desc()                          # radius 0: refused
    blobs = (lp.lf_blob * 1)()
    w = (C.c_float * lp.LF_POST_WEIGHTS)()
    yield lambda: lp.lf_render(0, views, 0, x, None)
    yield lambda: lp.lf_render(0, views, 0, A, x)
    yield lambda: lp.lf_render(0, views, 0, A, None, x)
    yield lambda: lp.lf_render_f16(0, views, 0, x, None)
    yield lambda: lp.lf_render_f16(0, views, 0, A, x)
    yield lambda: lp.lf_render_backward(0, views, 0, x, A)
    yield lambda: lp.lf_render_backward(0, views, 0, A, x)
    yield lambda: lp.lf_render_backward_idx(0, views, 0, A, x, A)
    yield lambda: lp.lf_render_backward_idx(0, views, 0, A, A, A, x)
    yield lambda: lp.lf_quantize_table(x, 0, 1, 4, 1, A, A)
    yield lambda: lp.lf_quantize_table(A, 0, 1, 4, 1, x, A)
    yield lambda: lp.lf_quantize_table(A, 0, 1, 4, 1, A, x)
    yield lambda: lp.lf_precompute_table(d, blobs, x)
    yield lambda: lp.lf_render_volume(d, blobs, views, 0, x)
    yield lambda: lp.lf_post_filter(0.0, (0, 0, 0), 3, w, views, 0, x, A)
    yield lambda: lp.lf_post_filter(0.0, (0, 0, 0), 3, w, views, 0, A, x)


@pytest.mark.parametrize("x", NOT_ADDRESSES, ids=lambda x: type(x).__name__)
def test_host_objects_are_not_device_addresses(x):
    for call in calls(x):
        with pytest.raises(TypeError):
            call()


def test_integers_and_none_reach_the_library():
    for x in (A, 0, None):
        for call in calls(x):
            with pytest.raises(lp.LfError):
                call()
