"""Catalogues around the sizes where the spatial sort changes its launches (a
block holds 1024 keys; up to 65536 keys a pass is one launch) and where a
count's tile pairs are taken in fewer parts: counts equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1208_3658_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_d,n_r", [(1, 1), (511, 512), (512, 512), (513, 512), (5, 16379),
                                     (16384, 16385), (32767, 32768), (32768, 32768),
                                     (32768, 32769)])
def test_wtheta_at_sort_sizes(n_d, n_r):
    from paper_1208_3658_gb300 import wtheta as W
    fp = synth.Patch(30.0, 8.0, 10.0, 18.0)
    D = O.radec_to_xyz(synth.clustered(fp, n_d, max(1, n_d // 50), 3.0, 3, "test", "data"))
    R = O.radec_to_xyz(synth.uniform(fp, n_r, 3, "test", "random"))
    e = W.wtheta_edges(1.0 / 60, 5.0, 12)
    c = torch.zeros(3 * (len(e) + 1), dtype=torch.int64, device="cuda")
    W.wtheta_count_wtheta(torch.from_numpy(D).cuda(), torch.from_numpy(R).cuda(), True, e, c)
    torch.cuda.synchronize()
    got = c.cpu().numpy().astype(np.uint64).reshape(3, -1)
    for g, (a, b, auto) in zip(got, ((D, None, True), (D, R, False), (R, None, True))):
        assert np.array_equal(g, O.count_xyz(a, b, e, auto))
