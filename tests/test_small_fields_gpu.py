"""Fields of a few arcsec with edges down to hundredths of an arcsec, where many
values of a step lie in guard bands (recount_band_values): counts equal the
oracle's, bit for bit."""
import numpy as np
import pytest

from oracle import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ARCSEC = 1.0 / 3600.0


def _field(n, side, seed):
    rng = np.random.default_rng(seed)
    p = np.stack([77.0 + side * rng.random(n), -41.0 + side * rng.random(n)], axis=1)
    return O.radec_to_xyz(p.reshape(-1))


@pytest.mark.parametrize("side", [0.3 * ARCSEC, 2 * ARCSEC, 36 * ARCSEC])
@pytest.mark.parametrize("lo,hi,K,linear", [(0.02 * ARCSEC, 10 * ARCSEC, 14, False),
                                            (0.0, 2 * ARCSEC, 5, True),
                                            (0.1 * ARCSEC, 0.2 * ARCSEC, 40, True)])
@pytest.mark.parametrize("n", [3001, 5000])
def test_counts_of_small_fields(n, lo, hi, K, linear, side):
    from paper_1208_3658_gb300 import wtheta as W
    e = W.wtheta_edges(lo, hi, K, W.BINS_LINEAR if linear else W.BINS_LN)
    A, B = _field(n, side, 1), _field(n - 700, side, 2)
    t = lambda x: None if x is None else torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    for a, b, auto in ((A, None, True), (A, B, False)):
        c = torch.zeros(K + 2, dtype=torch.int64, device="cuda")
        W.wtheta_count_xyz(t(a), t(b), e, auto, c)
        torch.cuda.synchronize()
        assert np.array_equal(c.cpu().numpy().astype(np.uint64), O.count_xyz(a, b, e, auto))
