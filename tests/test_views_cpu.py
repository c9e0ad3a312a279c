"""The binding's lf_view arrays (lumipath.make_views): the bytes that ctypes' own
field conversions give, and what those refuse stays refused."""
import ctypes as C
from types import SimpleNamespace

import numpy as np
import pytest

import lf_inputs
from paper_1903_03837_gb300 import lumipath as lp


def by_fields(views):
    arr = (lp.lf_view * len(views))()
    for a, v in zip(arr, views):
        a.eye[:], a.right[:], a.up[:], a.forward[:] = list(v.eye), list(v.right), list(v.up), list(v.forward)
        a.tan_half_x, a.tan_half_y = v.tan_half_x, v.tan_half_y
        a.width, a.height, a.out_offset = v.width, v.height, v.out_offset
    return arr


def view(**k):
    base = dict(eye=(1.1, 2.0, -3.0), right=(0.1, 0.2, 0.3), up=(4.0, 5.0, 6.0), forward=(7.0, 8.0, 9.0), tan_half_x=0.3,
                tan_half_y=0.2, width=640, height=480, out_offset=7)
    return SimpleNamespace(**{**base, **k})


@pytest.mark.parametrize("views", [
    lf_inputs.config_batching().views,
    [view(), view(eye=np.float32([1e-42, 0.1, -0.0]), up=np.float64([1e-50, 1 / 3, 1e30]), width=np.int64(3))],
    [view(eye=(1e39, float("nan"), float("-inf"))), view(height=-1), view(width=2**40 + 5), view(out_offset=2**63 + 1)],
])
def test_views_are_ctypes_own_bytes(views):
    assert bytes(lp.make_views(views)) == bytes(by_fields(views))
    assert C.sizeof(lp.lf_view) == 72


@pytest.mark.parametrize("bad,error", [(dict(eye=(1, 2)), ValueError), (dict(eye=(1, 2), right=(1, 2, 3, 4)), ValueError),
                                       (dict(width=None), TypeError), (dict(width=1.5), TypeError),
                                       (dict(tan_half_x="1"), TypeError)])
def test_views_that_are_refused(bad, error):
    with pytest.raises(error):
        lp.make_views([view(**bad)])
