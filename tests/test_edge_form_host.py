"""The edge jobs' decisions by host emulation of their FP32 steps (`span_emulation.py`,
no GPU): beyond the slack of an edge (`local_guard`) and of the chunk (`write_chunk`)
the sign of an edge job's value gives the side of the FP64 squared chord, for the
first and the second edge of a job (`two_edge_step`), near and far apart, with the
centres that `small_sphere` gives, and for points of A whose own chunk keeps the
origin as its centre (padding, or wider than 0.5)."""
import numpy as np
import pytest

import span_emulation as S
from host_calls import run

F = S.F


def test_slack_of_the_library(tmp_path):
    cs = [1e-10, 3.4e-9, 1e-6, 1e-3, 0.1, 1.0, 3.9, 4.0]
    out = run(tmp_path, "for (int i = 1; i < argc; ++i)"
                        ' printf("%.17g\\n", local_guard(atof(argv[i])));', [repr(c) for c in cs])
    got = np.array([float(x[0]) for x in out])
    assert np.allclose(got, S.local_guard(np.array(cs)), rtol=1e-13, atol=0)


@pytest.mark.parametrize("origin", [False, True])
@pytest.mark.parametrize("dev", [0.0, 4e-7])
@pytest.mark.parametrize("sep,size", [(3e-4, 1e-4), (3e-3, 1e-3), (0.02, 8e-3), (0.2, 7e-3),
                                      (0.2, 0.1), (1.0, 0.05), (1.9, 0.2), (1.99, 0.005)])
def test_sides_of_both_edges(sep, size, dev, origin):
    rng = np.random.default_rng([int(sep * 1e6), int(size * 1e6), int(dev * 1e9), origin])
    n = 250
    PA, PB = S.pairs_of_clouds(rng, n, sep, size, 32, 32)
    if dev:  # inputs normalised in FP32 are accepted
        PA = PA * (1 + dev * rng.uniform(-1, 1, (n, 1, 32)))
        PB = PB * (1 + dev * rng.uniform(-1, 1, (n, 1, 32)))
    ca, _, la, _, _, _ = S.write_chunk(PA, False, np.full(n, origin))
    assert np.all(ca == 0) == origin
    cb, rb, lb, kappa, hc, _ = S.write_chunk(PB, False)
    assert np.all((rb >= 0) & (rb <= 0.5))
    s = S.chord2(PA, PB)
    flat = s.reshape(n, -1)
    settled = total = tight = 0
    for k in range(12):
        # a first edge through the cloud of pairs (some on a pair's own value), and
        # a second one also in it, just above, or far above
        c = (flat[np.arange(n), rng.integers(0, 1024, n)] if k % 2
             else np.quantile(flat, rng.uniform(0, 1), axis=1))
        far = [np.quantile(flat, 0.9, axis=1), c * (1 + 1e-6), c + rng.uniform(0, 4, n),
               np.full(n, 4.0)][k % 4]
        c2 = np.minimum(np.maximum(far, c * (1 + 1e-7)), 4.0)
        ok = (c >= 1e-10) & (c2 > c)
        mid, mid2 = c.astype(F), c2.astype(F)
        for d, edge in zip(S.edge_values(la, ca, lb, cb, kappa, mid, mid2), (c, c2)):
            G = (np.array([S.half_slack(x) for x in edge]) + hc).astype(np.float64)[:, None, None]
            d = d.astype(np.float64)
            side = s < edge[:, None, None]
            sure = (np.abs(d) > G) & ok[:, None, None]
            assert np.array_equal((d < 0)[sure], side[sure])
            settled += int(sure.sum())
            total += int(ok.sum()) * 1024
            tight += int(((np.abs(d) > 0.02 * G) & ((d < 0) != side) & ok[:, None, None]).sum())
    # (unit vectors off by 4e-7 have a slack of their own size, 8e-7, which is more
    # than the squared chords of clouds 3e-4 apart: FP64 settles those)
    if 2 * np.median(hc) < 0.02 * np.median(np.ptp(flat, axis=1)):
        assert settled > 0.9 * total
    assert tight > 0 or sep < 1e-3   # a slack fifty times smaller would miscount
