"""Spans over any number of edges, against the oracle bit for bit: bin widths
from far above a group's span (no edge) to far below it (pair by pair), odd and
even numbers of edges, the diagonal tile pairs' own chunks, ragged last tiles,
and every histogram layout and tile size that takes spans."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1208_3658_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _points(n, seed):
    """Half uniform, half in clusters, in a 6 x 6 deg patch."""
    fp = synth.Patch(10.0, 6.0, -3.0, 3.0)
    a = synth.uniform(fp, n // 2, seed, "test", "random").reshape(-1, 2)
    b = synth.clustered(fp, n - n // 2, max(1, n // 100), 4.0, seed, "test", "data").reshape(-1, 2)
    return O.radec_to_xyz(np.concatenate([a, b]).reshape(-1))


@pytest.mark.parametrize("K", [1, 4, 13, 40, 256])
@pytest.mark.parametrize("n,tune", [(1500, None), (2305, dict(threads=64)),
                                    (3001, dict(threads=128)),
                                    (2049, dict(threads=128, hist_mode=4))])
def test_spans_of_many_edges(K, n, tune):
    from paper_1208_3658_gb300 import wtheta as W
    e = W.wtheta_edges(0.0, 8.0, K, W.BINS_LINEAR)
    A, B = _points(n, 5), _points(n - 333, 6)
    for a, b, auto in ((A, None, True), (A, B, False)):
        c = torch.zeros(K + 2, dtype=torch.int64, device="cuda")
        t = lambda x: None if x is None else torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
        if tune is None:
            W.wtheta_count_xyz(t(a), t(b), e, auto, c)
        else:
            W.wtheta_count_ex(t(a), t(b), True, e, auto, c, tune=tune)
        torch.cuda.synchronize()
        assert np.array_equal(c.cpu().numpy().astype(np.uint64), O.count_xyz(a, b, e, auto))
