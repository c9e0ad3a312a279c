"""The points within the filter kernel's radius (Section 2: a kernel of radius
sqrt(4 pi / n) around a hit, in units of the sphere's radius).

An image needs only the neighbours of nonzero weight, and the tent gives weight
0 at that radius and beyond. The render kernels therefore list the points within
the radius instead of ranking the nearest ones, which is the same image when the
points within it are among the 5 nearest (there are never more than 5), there is
always at least one, and the kernel tests every one of them: 7 lattice corners
from 8 continuous indices off a pole on, the 28 points nearest the pole up to
there. All of it is checked here by brute force: against a k-d tree over the FP64
points, with the lattice coordinates and the zone moved by more than their FP32
error as in the window study.
"""
import math

import numpy as np
import pytest

import oracle
from test_window_study import lattice_coords, points_and_tree, random_queries, window_candidates, window_corner

scipy_spatial = pytest.importorskip("scipy.spatial")

POLE = 8           # continuous-index distance from a pole below which the kernel scans
POLE_PTS = 28      # points scanned at a pole

# (du, dv) of the kernel's 7 corners in the quadrant's turned basis
CORNERS = np.array([(0, 0), (0, 1), (1, 0), (1, 1), (0, -1), (-1, 1), (-1, 0)], dtype=np.int32)


def sigma(n):
    return math.sqrt(4.0 * math.pi / n)


def pole_queries(rng, n, count):
    """Unit vectors within 33 continuous indices of either pole."""
    z = 1.0 - rng.uniform(0.0, min(2.0, 2 * 33 / n), count)
    ph = rng.uniform(0.0, 2 * np.pi, count)
    r = np.sqrt(np.maximum(0.0, 1.0 - z * z))
    return np.stack([np.cos(ph) * r, np.sin(ph) * r, np.where(rng.uniform(size=count) < 0.5, z, -z)], 1)


def pole_distance(q, n):
    """Continuous index counted from the nearer pole."""
    return (n * (1.0 - np.abs(q[:, 2])) - 1.0) * 0.5


@pytest.mark.parametrize("lo,hi,count", [(1, 130, 20_000), (130, 400, 8_000)])
def test_one_to_five_points_within_the_radius_small_sets(lo, hi, count):
    """Every n of the full scan and the first window sizes: 1 to 5 points lie
    within the radius, the 6th nearest at 1.04 radii or farther, the 5th within
    1.75, the nearest within 0.78."""
    rng = np.random.default_rng(lo)
    for n in range(lo, hi):
        tree = scipy_spatial.cKDTree(oracle.sf_points(n))
        q = np.concatenate([random_queries(rng, count), pole_queries(rng, n, count // 4)])
        d = tree.query(q, k=list(range(1, min(n, 6) + 1)))[0] / sigma(n)
        if n >= 6:
            assert d[:, 5].min() >= 1.04, n
        if n >= 5:
            assert d[:, 4].max() <= 1.75, n
        assert d[:, 0].max() <= 0.78, n


@pytest.mark.parametrize("n", [512, 997, 4096, 12288, 16384, 65536, 262144, 1 << 20, 1 << 24])
def test_one_to_five_points_within_the_radius(n):
    _, tree = points_and_tree(n)
    rng = np.random.default_rng(n + 1)
    q = np.concatenate([random_queries(rng, 400_000), pole_queries(rng, n, 100_000)])
    d = tree.query(q, k=[1, 5, 6], workers=-1)[0] / sigma(n)
    assert d[:, 0].max() <= 0.78 and d[:, 1].max() <= 1.75 and d[:, 2].min() >= 1.04


@pytest.mark.parametrize("n", [129, 200, 256, 1000, 4096, 16384, 65536, 262144, 1 << 20, 1 << 24])
def test_the_seven_corners_hold_every_point_within_the_radius(n):
    _, tree = points_and_tree(n)
    rng = np.random.default_rng(n + 2)
    q = np.concatenate([random_queries(rng, 500_000), pole_queries(rng, n, 100_000)])
    q = q[pole_distance(q, n) >= POLE - 1e-3]
    d, nn = tree.query(q, k=5, workers=-1)
    near = d < sigma(n) * (1.0 + 1e-4)       # FP32 rounding of the distance and the radius
    coords = lattice_coords(q, n)
    moves = [(a, b, 0.0) for a in (-2e-3, 0.0, 2e-3) for b in (-2e-3, 0.0, 2e-3)] + [(0.0, 0.0, -0.02), (0.0, 0.0, 0.02)]
    for du, dv, dk in moves:
        cand = window_candidates(window_corner(coords, du, dv, dk), CORNERS)
        for m in range(5):
            ok = ~near[:, m] | (cand == nn[:, m:m + 1]).any(axis=1)
            assert ok.all(), (n, du, dv, dk, m, int((~ok).sum()))


@pytest.mark.parametrize("n", [129, 200, 256, 1000, 4096, 65536, 1 << 24])
def test_the_pole_scan_holds_every_point_within_the_radius(n):
    _, tree = points_and_tree(n)
    q = pole_queries(np.random.default_rng(n + 3), n, 400_000)
    q = q[pole_distance(q, n) < POLE + 1e-3]
    assert len(q) > 10_000
    d, nn = tree.query(q, k=5, workers=-1)
    near = d < sigma(n) * (1.0 + 1e-4)
    from_pole = np.where(q[:, 2:] > 0, nn, n - 1 - nn)
    assert from_pole[near].max() < POLE_PTS


def test_the_corner_list_is_not_larger_than_needed():
    """Each of the 7 corners is the only one that holds some point within the
    radius (dropping any would lose points)."""
    n = 16384
    _, tree = points_and_tree(n)
    q = random_queries(np.random.default_rng(5), 400_000)
    q = q[pole_distance(q, n) >= POLE]
    d, nn = tree.query(q, k=5, workers=-1)
    near = d < sigma(n)
    cand = window_candidates(window_corner(lattice_coords(q, n), 0.0, 0.0, 0.0), CORNERS)
    for j in range(len(CORNERS)):
        assert (near & (nn == cand[:, j:j + 1])).any(), CORNERS[j]
