"""The builds without span code, one per tile size: auto and cross counts at the
edges of tiles and of an item's parts equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1208_3658_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [32, 64, 128])
@pytest.mark.parametrize("n", [2, 33, 255, 256, 257, 1025, 5000])
@pytest.mark.parametrize("hist_mode", [0, 3])
def test_no_span_builds(threads, n, hist_mode):
    from paper_1208_3658_gb300 import wtheta as W
    fp = synth.Patch(30.0, 8.0, 10.0, 18.0)
    A = O.radec_to_xyz(synth.clustered(fp, n, max(1, n // 50), 3.0, 3, "test", "data"))
    B = O.radec_to_xyz(synth.uniform(fp, n + 300, 3, "test", "random"))
    e = W.wtheta_edges(1.0 / 60, 5.0, 20)
    t = lambda x: None if x is None else torch.from_numpy(np.ascontiguousarray(x)).cuda()  # noqa: E731
    for a, b, auto in ((A, None, True), (A, B, False)):
        c = torch.zeros(len(e) + 1, dtype=torch.int64, device="cuda")
        W.wtheta_count_ex(t(a), t(b), True, e, auto, c,
                          tune=dict(threads=threads, hist_mode=hist_mode, span_bins=2))
        torch.cuda.synchronize()
        assert np.array_equal(c.cpu().numpy().astype(np.uint64), O.count_xyz(a, b, e, auto))
