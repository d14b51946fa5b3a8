"""The fitness kernel's large primitives: a row's covered columns from one
clamped floor per edge (clip_row in raster_dev.cuh), against the edge functions
evaluated at every pixel."""
import numpy as np
import pytest

W = 1280


def floor_div_clamped(n, d, cap, rel):
    """rel: error of the FP32 quotient (rcp.approx and three roundings stay within 2^-22)."""
    f = min(max(float(np.float32(n)) / d * (1.0 + rel), float(-cap - 1)), float(cap))
    q = int(np.floor(f))
    r = n - q * d
    return q - 1 if r < 0 else q + 1 if r >= d else q


def clip_row(p, q, i, lo, hi, rel):
    dx, dy = q[0] - p[0], q[1] - p[1]
    bias = 0 if dy < 0 or (dy == 0 and dx > 0) else 1
    e = dx * (256 * i - p[1]) - dy * (256 * lo - p[0]) - bias
    if dy == 0:
        return (lo, lo - 1) if dx != 0 and e < 0 else (lo, hi)
    f = floor_div_clamped(e >> 8, abs(dy), max(hi - lo + 1, 0), rel)
    return (lo, min(hi, lo + f)) if dy > 0 else (max(lo, lo - f), hi)


def covered(poly, i):
    """Columns of row i inside every edge, from the edge functions."""
    j = np.arange(W, dtype=object)
    on = np.ones(W, bool)
    for p, q in zip(poly, poly[1:] + poly[:1]):
        dx, dy = q[0] - p[0], q[1] - p[1]
        bias = 0 if dy < 0 or (dy == 0 and dx > 0) else 1
        on &= np.array(dx * (256 * i - p[1]) - dy * (256 * j - p[0]) - bias >= 0, bool)
    return on


def area2(a, b, c):
    return (b[0] - a[0]) * (c[1] - a[1]) - (c[0] - a[0]) * (b[1] - a[1])


@pytest.mark.parametrize("rel", [-2.0 ** -22, 0.0, 2.0 ** -22])
@pytest.mark.parametrize("reach", [40, 700, 16384])
def test_row_clip_equals_the_edge_functions(reach, rel):
    rng = np.random.default_rng(reach)
    for case in range(60):
        c = rng.integers(0, W, 2)
        poly = [tuple(int(v) for v in 256 * c + rng.integers(-256 * reach, 256 * reach + 1, 2)) for _ in range(3)]
        if case % 3 == 1:  # on the pixel lattice: edges through pixel centres
            poly = [(x & ~255, y & ~255) for x, y in poly]
        if case % 3 == 2:  # a horizontal edge through a row of centres
            poly[1] = (poly[1][0], poly[0][1] & ~255)
            poly[0] = (poly[0][0], poly[0][1] & ~255)
        A = area2(*poly)
        if A == 0:
            continue
        if A < 0:
            poly = [poly[0], poly[2], poly[1]]
        ys = [y for _, y in poly]
        rows = range(max(0, -(-min(ys) // 256)), min(1023, max(ys) // 256) + 1)
        for i in list(rows)[:: max(1, len(rows) // 12)]:
            lo, hi = max(0, -(-min(x for x, _ in poly) // 256)), min(W - 1, max(x for x, _ in poly) // 256)
            corners = poly + [poly[2]]  # a triangle repeats its last corner: an edge of no length
            for p, q in zip(corners, corners[1:] + corners[:1]):
                lo, hi = clip_row(p, q, i, lo, hi, rel)
            want = np.flatnonzero(covered(poly, i))
            got = np.arange(lo, hi + 1)
            assert np.array_equal(got, want), (poly, i, lo, hi)
