"""Soundness of the bounding spheres and of the intervals drawn from them, by host
emulation of their FP32 steps (`span_emulation.py`, no GPU): `small_sphere` around
8 and 32 points, `settle_chunks`' sphere around 8 chunk spheres, and `span_edges`'
interval, which has to hold every pair's FP64 squared chord."""
import numpy as np
import pytest

import span_emulation as S

F = S.F


def _inside(points, c, r):
    """FP64 distances of FP32 points (n, 3, k) from c, and whether r covers them."""
    d = points.astype(np.float64) - c.astype(np.float64)[:, :, None]
    return np.sqrt((d * d).sum(axis=1)) <= r.astype(np.float64)[:, None]


def _clouds(rng, n, size, k, kind):
    """n clouds of k unit vectors: uniform, clustered with an outlier, on a line,
    in two places, or one point k times."""
    c = S.unit(rng.normal(size=(n, 3)))[:, :, None]
    if kind == "uniform":
        t = size * rng.uniform(-1, 1, (n, 3, k))
    elif kind == "outlier":
        t = 0.01 * size * rng.normal(size=(n, 3, k))
        t[:, :, 0] *= 100
    elif kind == "line":
        t = size * rng.uniform(-1, 1, (n, 1, k)) * S.unit(rng.normal(size=(n, 3)))[:, :, None]
    elif kind == "two":
        t = size * np.where(np.arange(k) % 2, 1.0, -1.0) * S.unit(rng.normal(size=(n, 3)))[:, :, None]
        t = t + 1e-3 * size * rng.normal(size=(n, 3, k))
    else:
        t = np.zeros((n, 3, k))
    return S.unit(c + t)


KINDS = ["uniform", "outlier", "line", "two", "same"]


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("size", [1e-7, 1e-5, 1e-3, 0.05, 0.4])
def test_spheres_hold_their_points(size, kind, fused):
    rng = np.random.default_rng([int(size * 1e8), KINDS.index(kind), fused])
    for k in (8, 32):
        q = _clouds(rng, 1500, size, k, kind).astype(F)
        c, r = S.small_sphere(q, fused, 8 if k == 8 else 0)
        assert _inside(q, c, r).all()
        # no wider than the sphere around the mean of the box's ends
        mid = 0.5 * (q.min(axis=2) + q.max(axis=2)).astype(np.float64)
        far = np.sqrt(((q - mid[:, :, None]) ** 2).sum(axis=1).max(axis=1))
        assert np.all(r <= far * (1 + 1e-4) + 3e-7)
    # eight chunks of a sub-tile, apart from one another as well
    p = _clouds(rng, 1500, size, 256, kind)
    q = p.astype(F)
    spheres = [S.small_sphere(q[:, :, 32 * i:32 * i + 32], fused) for i in range(8)]
    c = np.stack([s[0] for s in spheres], axis=1)
    r = np.stack([s[1] for s in spheres], axis=1)
    g, R = S.sub_tile_sphere(c, r, fused)
    use = R < 3
    assert use.any() or size > 0.2
    assert _inside(q, g, R)[use].all()


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("kind", ["uniform", "outlier", "two"])
@pytest.mark.parametrize("s_a,s_b", [(1e-7, 1e-7), (3e-5, 1e-5), (2e-3, 5e-3), (0.05, 0.1),
                                     (0.3, 0.01)])
def test_every_pair_inside_the_interval(s_a, s_b, kind, fused):
    rng = np.random.default_rng([int(s_a * 1e8), int(s_b * 1e8), KINDS.index(kind), fused])
    n = 600
    B = _clouds(rng, n, s_b, 32, kind)
    # A: a sub-tile of 256 points at separations from coincident to antipodal
    sep = np.concatenate([np.zeros(60), 10.0 ** rng.uniform(-8, np.log10(2), n - 120),
                          2.0 - 10.0 ** rng.uniform(-8, -2, 60)])
    b0 = S.unit(B.mean(axis=2))
    t = rng.normal(size=(n, 3))
    t = S.unit(t - b0 * (b0 * t).sum(axis=1, keepdims=True))
    ang = 2 * np.arcsin(np.minimum(sep / 2, 1))[:, None]
    a0 = b0 * np.cos(ang) + t * np.sin(ang)
    A = S.unit(a0[:, :, None] + s_a * rng.uniform(-1, 1, (n, 3, 256)))
    a32, b32 = A.astype(F), B.astype(F)
    cb, rb = S.small_sphere(b32, fused)
    s = S.chord2(A, B)

    def check(ca, ra, lo, hi, use):
        slo, shi = S.span_interval(ca, ra, cb, rb, fused)
        part = s[:, lo:hi][use]
        assert np.all(part >= slo.astype(np.float64)[use, None, None])
        assert np.all(part <= shi.astype(np.float64)[use, None, None])

    for g in range(0, 32, 5):
        ca, ra = S.small_sphere(a32[:, :, 8 * g:8 * g + 8], fused, 8 * (g % 4))
        check(ca, ra, 8 * g, 8 * g + 8, np.ones(n, bool))
    spheres = [S.small_sphere(a32[:, :, 32 * i:32 * i + 32], fused) for i in range(8)]
    c = np.stack([x[0] for x in spheres], axis=1)
    r = np.stack([x[1] for x in spheres], axis=1)
    g, R = S.sub_tile_sphere(c, r, fused)
    check(g, R, 0, 256, R < 3)


def test_a_sphere_without_its_slack_would_not_do():
    """The emulation sees a missing slack: radii a millionth too small leave points
    outside, and an interval without its absolute term leaves pairs outside."""
    rng = np.random.default_rng(3)
    q = _clouds(rng, 4000, 1e-3, 32, "uniform").astype(F)
    c, r = S.small_sphere(q, False)
    assert not _inside(q, c, (r * F(1 - 1.2e-6)).astype(F)).all()
    A, B = S.pairs_of_clouds(rng, 4000, 0.3, 0.0, 8, 32)
    ca, ra = S.small_sphere(A.astype(F), False)
    cb, rb = S.small_sphere(B.astype(F), False)
    s = S.chord2(A, B)
    d = (ca - cb).astype(np.float64)
    exact = (d * d).sum(axis=1)[:, None, None]     # (both radii are zero here)
    assert np.any(np.abs(s - exact) > 1e-9)
