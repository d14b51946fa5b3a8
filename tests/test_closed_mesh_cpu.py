"""The rule by which the fitness kernel draws a closed mesh by its front faces
alone, checked on the CPU against the oracle's union of all faces.

When every edge of a mesh is traversed equally often in both directions, the
triangles that cover a pixel centre under the top-left rule have as many positive
as negative orientations among them (the signed count is the winding number of
a closed chain), so the triangles of one orientation cover the silhouette.
That holds for any snapped corners -- also folded, degenerate or coinciding
ones -- as long as no triangle is dropped for a flagged corner.
"""
import numpy as np
import pytest

import oracle
from paper_2603_11404_gb300 import workload as wl


def _both(snap, tris, W, H):
    flag = np.zeros(len(snap), np.uint8)
    full = oracle.raster(snap, flag, tris, W, H)[0]
    front = oracle.raster(snap, flag, tris, W, H, True)[0]
    back = oracle.raster(snap, flag, tris[:, ::-1], W, H, True)[0]  # the other orientation
    return full, front, back


@pytest.mark.parametrize("size", ["c1", "800"])
def test_front_faces_cover_the_instrument(size):
    sc = wl.make_scene(size, "c1")
    _, tris, _ = sc.flat()
    rng = np.random.default_rng(7)
    drawn = 0
    for _ in range(12):
        pr = oracle.project(sc, wl.sample_state(rng, sc.K))
        if pr["flag"].any():
            continue
        full, front, back = _both(pr["snap"], tris, sc.K.width, sc.K.height)
        assert np.array_equal(full, front) and np.array_equal(full, back)
        drawn += int(full.any())
    assert drawn > 5


def _closed(kind, rng):
    if kind == "tetrahedron":
        return 4, np.array([[0, 1, 2], [0, 3, 1], [1, 3, 2], [2, 3, 0]], np.int32)
    n, m = int(rng.integers(3, 7)), int(rng.integers(3, 7))  # a torus of n x m quads
    q = lambda i, j: (i % n) * m + j % m
    t = []
    for i in range(n):
        for j in range(m):
            t += [[q(i, j), q(i + 1, j), q(i + 1, j + 1)], [q(i, j), q(i + 1, j + 1), q(i, j + 1)]]
    return n * m, np.array(t, np.int32)


@pytest.mark.parametrize("kind", ["tetrahedron", "torus"])
@pytest.mark.parametrize("step", [1, 128, 256])
def test_any_corners_of_a_closed_mesh(kind, step):
    """Random corners, free or on half and whole pixels (edges through centres,
    coinciding and collinear corners), partly outside the image."""
    rng = np.random.default_rng(31 + step)
    W = H = 24
    for _ in range(60):
        nv, tris = _closed(kind, rng)
        snap = rng.integers(-6 * 256 // step, 30 * 256 // step, (nv, 2)).astype(np.int64) * step
        full, front, back = _both(snap, tris, W, H)
        assert np.array_equal(full, front) and np.array_equal(full, back)


def test_an_open_mesh_needs_both_sides():
    """The rule is not vacuous: without one face the front faces are not enough."""
    rng = np.random.default_rng(5)
    differs = 0
    for _ in range(40):
        nv, tris = _closed("tetrahedron", rng)
        snap = rng.integers(0, 24 * 256, (nv, 2)).astype(np.int64)
        full, front, back = _both(snap, tris[1:], 24, 24)
        differs += int(not np.array_equal(full, front) or not np.array_equal(full, back))
    assert differs > 10
