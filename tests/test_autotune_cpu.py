"""The autotuner's candidates: launches the library accepts, each different from the
others (the persistent flag changes no launch)."""
from paper_1903_03837_gb300 import autotune


def test_no_two_candidates_are_the_same_launch():
    for cands in (autotune.CANDIDATES, autotune.QUICK):
        shapes = [c[:4] for c in cands]
        assert len(set(shapes)) == len(shapes)
    assert set(autotune.QUICK) <= set(autotune.CANDIDATES)


def test_candidates_are_valid_shapes():
    for tw, th, ww, order, persistent in autotune.CANDIDATES:
        assert tw * th <= 256 and tw % ww == 0 and th % (32 // ww) == 0 and order in (0, 1) and persistent in (0, 1)
        L = autotune.as_launch((tw, th, ww, order, persistent))
        assert set(L) == {"tile_w", "tile_h", "warp_w", "order", "persistent", "ctas_per_sm"}
