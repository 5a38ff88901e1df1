"""Soundness of the span jobs' local form, by host emulation (no GPU).

A two- or three-slot job decides each pair by the sign of
d = (s - mid) / 2 = A0 - a.b', computed in FP32 from coordinates relative to
the centres of the points' own chunks (`write_chunk`, `recentre`, `span_part`,
`two_slot_step`).  The decision counts only if |d| exceeds half the edge's slack
(`local_guard`) plus half the chunk's (`write_chunk`).  The test evaluates the
same FP32 steps in numpy and checks that every pair beyond the slack lies on
that side in the FP64 predicate, that the slack is what the derivation gives
(not looser than 2.5e-7 at ordinary sizes), and that a fiftieth of it would not do."""
import numpy as np
import pytest

F = np.float32
U = 2.0 ** -24


def _fma(a, b, c):
    """fl32(a b + c): exact product in FP64; the second rounding can differ
    from a true fma by an FP32 ulp only in halfway cases."""
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def _edge_slack(c):
    """local_guard: 1.05 u (2 sqrt(c) + 16 c) + 1e-13, halved and rounded up."""
    g = 0.5 * (1.05 * U * (2.0 * np.sqrt(c) + 16.0 * c) + 1e-13)
    return np.nextafter(F(g), F(np.inf))


def _chunk(p):
    """write_chunk for p (3, 32) FP64: centre, local coordinates, kappa, half slack."""
    p32 = p.astype(F)
    c = (p32.astype(np.float64).sum(axis=1) / 32).astype(F)
    r = F(np.sqrt(((p32 - c[:, None]).astype(np.float64) ** 2).sum(axis=0).max()) * (1 + 1e-6))
    c64 = c.astype(np.float64)
    loc = (p - c64[:, None]).astype(F)
    kb = ((p - c64[:, None]) * (p + c64[:, None])).sum(axis=0)
    kappa = F(0.5 * (kb.min() + kb.max()))
    dev = max(kb.max() - float(kappa), float(kappa) - kb.min())
    rr = float(r) + 2.4e-7
    slack = 1.05 * (dev + U * (12 * rr + 80 * rr * rr + 5 * abs(float(kappa))))
    return c, loc, r, kappa, F(0.5 * slack)


def _unit_cluster(rng, centre, size, n):
    v = centre[:, None] + size * rng.uniform(-1, 1, (3, n))
    return v / np.sqrt((v * v).sum(axis=0))


def _rot(rng):
    q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
    return q


def _decide(A, ca, B, cb, kappa, mid):
    """d for the pairs (a, b) of local coordinates A (3, na) and B (3, nb)."""
    D = (ca - cb).astype(F)
    lx = (A + D[:, None]).astype(F)
    ab = (A + ca[:, None]).astype(F)
    km = F(kappa - mid)
    t = _fma(lx[2], lx[2], np.full(lx.shape[1], km, F))
    t = _fma(lx[0], lx[0], _fma(lx[1], lx[1], t))
    a0 = (F(0.5) * t).astype(F)[:, None]
    d = _fma(ab[2][:, None], -B[2][None, :], np.broadcast_to(a0, (A.shape[1], B.shape[1])))
    return _fma(ab[0][:, None], -B[0][None, :], _fma(ab[1][:, None], -B[1][None, :], d))


@pytest.mark.parametrize("sep,size,dev", [
    (3e-4, 1e-4, 0.0), (3e-3, 1e-3, 0.0), (0.02, 8e-3, 0.0), (0.2, 7e-3, 0.0), (0.2, 0.1, 0.0),
    (1.0, 0.05, 0.0), (1.9, 0.2, 0.0), (0.2, 7e-3, 4e-7), (0.02, 8e-3, 4e-7)])
def test_decisions_match_fp64(sep, size, dev):
    """sep: chord between the clusters; dev: deviation of |b| from 1 (inputs
    normalised in FP32 are accepted)."""
    rng = np.random.default_rng([int(sep * 1e6), int(size * 1e6), int(dev * 1e9)])
    settled = wrong_if_smaller = total = 0
    for _ in range(60):
        R = _rot(rng)
        ang = 2 * np.arcsin(sep / 2)
        a0 = R @ np.array([1.0, 0, 0])
        b0 = R @ np.array([np.cos(ang), np.sin(ang), 0])
        PA, PB = _unit_cluster(rng, a0, size, 32), _unit_cluster(rng, b0, size, 32)
        if dev:
            PB = PB * (1 + dev * rng.uniform(-1, 1, 32))
        ca, la, ra, _, _ = _chunk(PA)
        cb, lb, rb, kappa, hc = _chunk(PB)
        assert rb <= 0.5
        dx = PA[:, :, None] - PB[:, None, :]
        s = (dx[0] * dx[0] + dx[1] * dx[1]) + dx[2] * dx[2]
        # edges through the cloud of pairs, some exactly on a pair's value
        for c in np.concatenate([rng.choice(s.ravel(), 6), np.quantile(s, [0.1, 0.5, 0.9])]):
            if c < 1e-10:
                continue
            mid, G = F(c), float(_edge_slack(c)) + float(hc)
            d = _decide(la, ca, lb, cb, kappa, mid).astype(np.float64)
            sure = np.abs(d) > G
            assert np.array_equal((d < 0)[sure], (s < c)[sure])
            settled += int(sure.sum())
            total += s.size
            wrong_if_smaller += int(((np.abs(d) > 0.02 * G) & ((d < 0) != (s < c))).sum())
            if not dev and sep <= 0.2 and size <= 8e-3:
                assert G < 2.5e-7
    assert settled > 0.9 * total
    assert wrong_if_smaller > 0 or sep < 1e-3  # a slack fifty times smaller would miscount


