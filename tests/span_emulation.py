"""The pair kernel's FP32 sphere and edge arithmetic, step by step in numpy, for
the host tests of its bounds: bounding spheres (`small_sphere`), a chunk's local
coordinates, kappa and slack (`write_chunk`), the sphere of a sub-tile's chunks
(`settle_chunks`), the interval of a span (`span_edges`) and the values an edge
job decides by (`recentre`, `span_part`, `two_edge_step`).  Arrays carry the
configurations first, then the coordinate, then the point.  fused: products
contracted into the sums, where the compiler may do so."""
import numpy as np

F = np.float32
U = 2.0 ** -24


def fma(a, b, c):
    """fl32(a b + c): exact product in FP64; the FP64 sum's rounding can differ
    from a true fma by an FP32 ulp only in halfway cases."""
    return (np.asarray(a, np.float64) * np.asarray(b, np.float64)
            + np.asarray(c, np.float64)).astype(F)


def norm2(d, fused):
    """dx dx + dy dy + dz dz of d (n, 3, ...)."""
    x, y, z = d[:, 0], d[:, 1], d[:, 2]
    if fused:
        return fma(z, z, fma(y, y, (x * x).astype(F)))
    return (((x * x).astype(F) + (y * y).astype(F)).astype(F) + (z * z).astype(F)).astype(F)


def small_sphere(P, fused, first_lane=0):
    """P (n, 3, W) FP32: centre (n, 3) and radius (n)."""
    lo, hi = P.min(axis=2), P.max(axis=2)
    c = (F(0.5) * (lo + hi).astype(F)).astype(F)
    b = c.copy()
    best = np.full(len(P), np.inf, F)
    lane = np.arange(P.shape[2], dtype=np.uint32) + np.uint32(first_lane)
    rows = np.arange(len(P))
    for it in range(9):
        d2 = norm2((P - c[:, :, None]).astype(F), fused)
        key = (d2.view(np.uint32) & ~np.uint32(31)) | lane
        far = key.argmax(axis=1)
        m = (key.max(axis=1) & ~np.uint32(31)).view(F)
        better = m < best
        best = np.where(better, m, best)
        b[better] = c[better]
        st = F(1.0) / F(it + 3)
        step = (P[rows, :, far] - c).astype(F)
        c = fma(st, step, c) if fused else (c + (st * step).astype(F)).astype(F)
    r2 = norm2((P - b[:, :, None]).astype(F), fused).max(axis=1)
    return b, (np.sqrt(r2) * F(1.0 + F(1e-6))).astype(F)


def write_chunk(p, fused, pad=None):
    """p (n, 3, 32) FP64; pad (n): the chunk holds padding (only its centre and
    radius show it).  Returns centre, radius (-1 padded, 3 wide), local
    coordinates, kappa, half the slack, and the four groups' spheres."""
    q = p.astype(F)
    pad = np.zeros(len(p), bool) if pad is None else pad
    groups = [small_sphere(q[:, :, 8 * g:8 * g + 8], fused, 8 * g) for g in range(4)]
    c, r = small_sphere(q, fused)
    wide = ~(r <= F(0.5))
    c = np.where((pad | wide)[:, None], F(0), c)
    c64 = c.astype(np.float64)[:, :, None]
    e = p - c64
    loc = e.astype(F)
    k = e * (p + c64)
    kb = (k[:, 0] + k[:, 1]) + k[:, 2]
    kappa = (0.5 * (kb.min(axis=1) + kb.max(axis=1))).astype(F)
    k64 = kappa.astype(np.float64)
    dev = np.maximum(kb.max(axis=1) - k64, k64 - kb.min(axis=1)).astype(F)
    rr = r + F(2.4e-7)
    slack = F(1.05) * (dev + F(5.9604645e-8) * (F(12) * rr + F(80) * rr * rr
                                                + F(5) * np.abs(kappa)))
    radius = np.where(pad, F(-1), np.where(wide, F(3), r))
    return c, radius, loc, kappa, (F(0.5) * slack).astype(F), groups


def local_guard(c):
    """The slack of s - mid around an edge c, less the chunk's part (FP64)."""
    return 1.05 * U * (2.0 * np.sqrt(c) + 16.0 * c) + 1e-13


def half_slack(c):
    """An edge's table entry: half of local_guard, rounded up to FP32."""
    x = 0.5 * local_guard(c)
    f = F(x)
    return f if float(f) >= x else np.nextafter(f, F(np.inf))


def edge_values(A, ca, B, cb, kappa, mid, mid2):
    """d of every pair for the edge mid, and for the second edge mid2 of a job:
    A (n, 3, na) and B (n, 3, nb) local to ca and cb (n, 3)."""
    D = (ca - cb).astype(F)
    lx = (A + D[:, :, None]).astype(F)
    ax = (A + ca[:, :, None]).astype(F)
    km = (kappa - mid).astype(F)[:, None]
    t = fma(lx[:, 2], lx[:, 2], km)
    t = fma(lx[:, 0], lx[:, 0], fma(lx[:, 1], lx[:, 1], t))
    a0 = (F(0.5) * t).astype(F)[:, :, None]
    b = -B[:, :, None, :]
    a = ax[:, :, :, None]
    d = fma(a[:, 0], b[:, 0], fma(a[:, 1], b[:, 1], fma(a[:, 2], b[:, 2], a0)))
    ndel = (F(0.5) * (mid - mid2).astype(F)).astype(F)[:, None, None]
    return d, (d + ndel).astype(F)


def span_interval(ca, ra, cb, rb, fused):
    """span_edges' [slo, shi]."""
    d = (ca - cb).astype(F)
    # sqrt.approx.f32 is within 2^-22 of the root: both ends of that
    root = np.sqrt(norm2(d, fused).astype(np.float64))
    k1, k2 = F(1.0 + F(1e-6)), F(1.0 - F(1e-6))
    w = (ra + rb).astype(F)
    slo = shi = None
    for e in (-1.0, 1.0):
        dc = (root * (1.0 + e * 2.0 ** -22)).astype(F)
        if fused:
            rr = fma(w, k1, F(1e-6))
            lo, hi = fma(dc, k2, -rr), fma(dc, k1, rr)
        else:
            rr = ((w * k1).astype(F) + F(1e-6)).astype(F)
            lo, hi = ((dc * k2).astype(F) - rr).astype(F), ((dc * k1).astype(F) + rr).astype(F)
        lo = np.maximum(lo, F(0))
        a = ((lo * lo).astype(F) * F(1.0 - F(1e-5))).astype(F)
        b = ((hi * hi).astype(F) * F(1.0 + F(1e-5))).astype(F)
        # the worse of the two: the interval has to hold with either
        slo = a if slo is None else np.maximum(slo, a)
        shi = b if shi is None else np.minimum(shi, b)
    return slo, shi


def sub_tile_sphere(c, r, fused):
    """settle_chunks' sphere around 8 chunk spheres: c (n, 8, 3), r (n, 8)."""
    s = c.copy()
    for o in (1, 2, 4):
        s = (s + s[:, np.arange(8) ^ o]).astype(F)
    g = (s * F(0.125)).astype(F)             # (sums commute: the same in every lane)
    d = (c - g).astype(F)
    root = np.sqrt(norm2(np.moveaxis(d, 2, 1), fused).astype(np.float64))
    dist = (root * (1.0 - 2.0 ** -22)).astype(F)
    w = (dist + r).astype(F)
    k = F(1.0 + F(4e-6))
    rad = fma(w, k, F(2e-7)) if fused else ((w * k).astype(F) + F(2e-7)).astype(F)
    rad = np.where((r >= 0) & (r <= F(0.5)), rad, F(3))
    return g[:, 0], rad.max(axis=1)


def chord2(A, B):
    """The FP64 squared chords of A (n, 3, na) and B (n, 3, nb)."""
    d = A[:, :, :, None] - B[:, :, None, :]
    return (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]


def unit(v, axis=1):
    return v / np.sqrt((v * v).sum(axis=axis, keepdims=True))


def pairs_of_clouds(rng, n, sep, size, na, nb):
    """Two clouds of unit vectors about sep (chord) apart, anywhere on the sphere."""
    a0 = unit(rng.normal(size=(n, 3)))
    t = rng.normal(size=(n, 3))
    t = unit(t - a0 * (a0 * t).sum(axis=1, keepdims=True))
    ang = 2.0 * np.arcsin(np.minimum(np.asarray(sep, np.float64) / 2.0, 1.0))
    ang = np.broadcast_to(ang, (n,))[:, None]
    b0 = a0 * np.cos(ang) + t * np.sin(ang)
    size = np.broadcast_to(np.asarray(size, np.float64), (n,))[:, None, None]
    cloud = lambda m, k: unit(m[:, :, None] + size * rng.uniform(-1, 1, (n, 3, k)))  # noqa: E731
    return cloud(a0, na), cloud(b0, nb)
